// Instantiations of the strip-chain polynomial-interpolation forward wavefront (float cell updates), orders 12..12 (one unit per group of orders so that the units compile in parallel).
#include "sk_fwd_chain.cuh"
#include "sk_dispatch.h"

namespace sk {

const void* fwd_interp_chain_ptr_f32_4(int N) {
    switch (N) {
        case 12: return reinterpret_cast<const void*>(&fwd_chain_kernel<float, 12, 12 + sk::kJF32, true>);
        default: return nullptr;
    }
}

}  // namespace sk
