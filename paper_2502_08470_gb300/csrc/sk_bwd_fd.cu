// Instantiations of the finite-difference adjoint from the forward tape (dyadic orders 0..4).
#include "sk_bwd_fd.cuh"
#include "sk_dispatch.h"

namespace sk {

namespace {
template <typename T, int ORDER, bool NARROW = false>
const void* bwd_fd_rows(int lam) {
    if constexpr (NARROW) {  // one refined column a step (fd_narrow)
        switch (lam) {
            case 1: return reinterpret_cast<const void*>(&bwd_fd_tape_kernel<T, ORDER, 2, 1>);
            case 2: return reinterpret_cast<const void*>(&bwd_fd_tape_kernel<T, ORDER, 4, 1>);
            case 3: return reinterpret_cast<const void*>(&bwd_fd_tape_kernel<T, ORDER, 8, 1>);
            case 4: return reinterpret_cast<const void*>(&bwd_fd_tape_kernel<T, ORDER, 16, 1>);
            default: return nullptr;
        }
    }
    switch (lam) {
        case 0: return reinterpret_cast<const void*>(&bwd_fd_tape_kernel<T, ORDER, 1>);
        case 1: return reinterpret_cast<const void*>(&bwd_fd_tape_kernel<T, ORDER, 2>);
        case 2: return reinterpret_cast<const void*>(&bwd_fd_tape_kernel<T, ORDER, 4>);
        case 3: return reinterpret_cast<const void*>(&bwd_fd_tape_kernel<T, ORDER, 8>);
        case 4: return reinterpret_cast<const void*>(&bwd_fd_tape_kernel<T, ORDER, 16>);
        default: return nullptr;
    }
}
}  // namespace

const void* bwd_fd_tape_ptr(int T, int order, int lam, bool narrow) {
    if (narrow)  // FP64
        return order == 3 ? bwd_fd_rows<double, 3, true>(lam) : order == 2 ? bwd_fd_rows<double, 2, true>(lam) : bwd_fd_rows<double, 1, true>(lam);
    if (T == 1) return order == 3 ? bwd_fd_rows<float, 3>(lam) : order == 2 ? bwd_fd_rows<float, 2>(lam) : bwd_fd_rows<float, 1>(lam);
    return order == 3 ? bwd_fd_rows<double, 3>(lam) : order == 2 ? bwd_fd_rows<double, 2>(lam) : bwd_fd_rows<double, 1>(lam);
}

int fd_tape_row_elems(int T, int lam, bool narrow) {
    const int C = fd_tape_cols(lam, narrow);
    return T ? fd_tape_row<float>(1 << lam, C) : fd_tape_row<double>(1 << lam, C);
}

int fd_tape_cols(int lam, bool narrow) { return narrow ? 1 : fd_cols(1 << lam); }

int bwd_fd_ring_bytes(int T, int lam, bool narrow) {
    if (narrow) {  // FP64
        switch (lam) {
            case 1: return fd_ring_warp_bytes<double, 2, 1>();
            case 2: return fd_ring_warp_bytes<double, 4, 1>();
            case 3: return fd_ring_warp_bytes<double, 8, 1>();
            case 4: return fd_ring_warp_bytes<double, 16, 1>();
            default: return 0;
        }
    }
    switch (lam) {
        case 0: return T ? fd_ring_warp_bytes<float, 1>() : fd_ring_warp_bytes<double, 1>();
        case 1: return T ? fd_ring_warp_bytes<float, 2>() : fd_ring_warp_bytes<double, 2>();
        case 2: return T ? fd_ring_warp_bytes<float, 4>() : fd_ring_warp_bytes<double, 4>();
        case 3: return T ? fd_ring_warp_bytes<float, 8>() : fd_ring_warp_bytes<double, 8>();
        case 4: return T ? fd_ring_warp_bytes<float, 16>() : fd_ring_warp_bytes<double, 16>();
        default: return 0;
    }
}

}  // namespace sk
