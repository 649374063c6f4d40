// Instantiations of the strip-chain polynomial-interpolation forward wavefront (double cell updates), orders 9..10 (one unit per group of orders so that the units compile in parallel).
#include "sk_fwd_chain.cuh"
#include "sk_dispatch.h"

namespace sk {

const void* fwd_interp_chain_ptr_f64_2(int N) {
    switch (N) {
        case 9: return reinterpret_cast<const void*>(&fwd_chain_kernel<double, 9, 9 + sk::kJF64, true>);
        case 10: return reinterpret_cast<const void*>(&fwd_chain_kernel<double, 10, 10 + sk::kJF64, true>);
        default: return nullptr;
    }
}

}  // namespace sk
