// Instantiations of the strip-chain approximation forward wavefront that records the tape of output
// derivatives (double cell updates; the orders the tape adjoint supports).
#include "sk_fwd_chain.cuh"
#include "sk_dispatch.h"

namespace sk {

namespace {
template <int N>
const void* kernel() {
    return reinterpret_cast<const void*>(&fwd_chain_kernel<double, N, N, false, true>);
}
}  // namespace

const void* fwd_approx_chain_tape_ptr_f64(int N) {
    switch (N) {
        case 2: return kernel<2>();
        case 3: return kernel<3>();
        case 4: return kernel<4>();
        case 5: return kernel<5>();
        case 6: return kernel<6>();
        case 7: return kernel<7>();
        case 8: return kernel<8>();
        case 9: return kernel<9>();
        case 10: return kernel<10>();
        case 12: return kernel<12>();
        default: return nullptr;
    }
}

}  // namespace sk
