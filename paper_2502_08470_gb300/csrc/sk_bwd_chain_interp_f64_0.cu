// Instantiations of the strip-chain tape adjoint of the interpolation scheme, orders 2..8 (double cell updates).
#include "sk_bwd_chain.cuh"
#include "sk_dispatch.h"

namespace sk {

const void* bwd_chain_interp_ptr_f64_0(int N) {
    switch (N) {
        case 2: return reinterpret_cast<const void*>(&bwd_chain_kernel<double, 2, true>);
        case 3: return reinterpret_cast<const void*>(&bwd_chain_kernel<double, 3, true>);
        case 4: return reinterpret_cast<const void*>(&bwd_chain_kernel<double, 4, true>);
        case 5: return reinterpret_cast<const void*>(&bwd_chain_kernel<double, 5, true>);
        case 6: return reinterpret_cast<const void*>(&bwd_chain_kernel<double, 6, true>);
        case 7: return reinterpret_cast<const void*>(&bwd_chain_kernel<double, 7, true>);
        case 8: return reinterpret_cast<const void*>(&bwd_chain_kernel<double, 8, true>);
        default: return nullptr;
    }
}

}  // namespace sk
