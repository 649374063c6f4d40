// Instantiations of the strip-chain tape adjoint of the approximation scheme (float cell updates).
#include "sk_bwd_chain.cuh"
#include "sk_dispatch.h"

namespace sk {

const void* bwd_chain_approx_ptr_f32(int N) {
    switch (N) {
        case 2: return reinterpret_cast<const void*>(&bwd_chain_kernel<float, 2, false>);
        case 3: return reinterpret_cast<const void*>(&bwd_chain_kernel<float, 3, false>);
        case 4: return reinterpret_cast<const void*>(&bwd_chain_kernel<float, 4, false>);
        case 5: return reinterpret_cast<const void*>(&bwd_chain_kernel<float, 5, false>);
        case 6: return reinterpret_cast<const void*>(&bwd_chain_kernel<float, 6, false>);
        case 7: return reinterpret_cast<const void*>(&bwd_chain_kernel<float, 7, false>);
        case 8: return reinterpret_cast<const void*>(&bwd_chain_kernel<float, 8, false>);
        case 9: return reinterpret_cast<const void*>(&bwd_chain_kernel<float, 9, false>);
        case 10: return reinterpret_cast<const void*>(&bwd_chain_kernel<float, 10, false>);
        case 12: return reinterpret_cast<const void*>(&bwd_chain_kernel<float, 12, false>);
        default: return nullptr;
    }
}

}  // namespace sk
