// Instantiations of the polynomial-interpolation forward wavefront (double cell updates), orders 2..6 (one unit per group of orders so that the units compile in parallel).
#include "sk_fwd_poly.cuh"
#include "sk_dispatch.h"

namespace sk {

const void* fwd_interp_ptr_f64_0(int N) {
    switch (N) {
        case 2: return reinterpret_cast<const void*>(&fwd_poly_kernel<double, 2, 2 + sk::kJF64, true, false>);
        case 3: return reinterpret_cast<const void*>(&fwd_poly_kernel<double, 3, 3 + sk::kJF64, true, false>);
        case 4: return reinterpret_cast<const void*>(&fwd_poly_kernel<double, 4, 4 + sk::kJF64, true, false>);
        case 5: return reinterpret_cast<const void*>(&fwd_poly_kernel<double, 5, 5 + sk::kJF64, true, false>);
        case 6: return reinterpret_cast<const void*>(&fwd_poly_kernel<double, 6, 6 + sk::kJF64, true, false>);
        default: return nullptr;
    }
}

}  // namespace sk
