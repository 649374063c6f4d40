// Instantiations of the strip-chain tape adjoint of the interpolation scheme, orders 9..12 (double cell updates).
#include "sk_bwd_chain.cuh"
#include "sk_dispatch.h"

namespace sk {

const void* bwd_chain_interp_ptr_f64_1(int N) {
    switch (N) {
        case 9: return reinterpret_cast<const void*>(&bwd_chain_kernel<double, 9, true>);
        case 10: return reinterpret_cast<const void*>(&bwd_chain_kernel<double, 10, true>);
        case 11: return reinterpret_cast<const void*>(&bwd_chain_kernel<double, 11, true>);
        case 12: return reinterpret_cast<const void*>(&bwd_chain_kernel<double, 12, true>);
        default: return nullptr;
    }
}

const void* bwd_chain_ptr(int T, int N, bool interp) {
    if (T == 1) return interp ? bwd_chain_interp_ptr_f32(N) : bwd_chain_approx_ptr_f32(N);
    if (!interp) return bwd_chain_approx_ptr_f64(N);
    const void* k = bwd_chain_interp_ptr_f64_0(N);
    return k ? k : bwd_chain_interp_ptr_f64_1(N);
}

}  // namespace sk
