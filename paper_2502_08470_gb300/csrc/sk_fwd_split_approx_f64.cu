// Instantiations of the approximation forward wavefront whose cells are split over four warps (FP64).
#include "sk_fwd_split.cuh"
#include "sk_dispatch.h"

namespace sk {

const void* fwd_split_interp_ptr_f64(int N);

namespace {
template <int N>
const void* kernel() {
    return reinterpret_cast<const void*>(&fwd_split_kernel<N, N, false>);
}
}  // namespace

const void* fwd_split_ptr_f64(bool interp, int N) {
    if (interp) return fwd_split_interp_ptr_f64(N);
    switch (N) {
        case 2: return kernel<2>();
        case 3: return kernel<3>();
        case 4: return kernel<4>();
        case 5: return kernel<5>();
        case 6: return kernel<6>();
        case 7: return kernel<7>();
        case 8: return kernel<8>();
        default: return nullptr;
    }
}

}  // namespace sk
