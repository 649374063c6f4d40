// Instantiations of the finite-difference forward wavefront and the kernel lookup.
#include <algorithm>

#include "sk_dispatch.h"
#include "sk_fwd_fd.cuh"

namespace sk {

namespace {
template <typename T, int ORDER>
const void* fd_rows(int lam, bool loop = false) {
    if constexpr (sizeof(T) == 4)
        if (loop && lam == 0) return reinterpret_cast<const void*>(&fwd_fd_kernel<T, ORDER, 1, 1, false, 1, true>);
    // rows per lane: R = min(2^lambda, 16) (a divisor of 2^lambda, so a lane's rows share a cell)
    switch (lam < 4 ? lam : 4) {
        case 0: return reinterpret_cast<const void*>(&fwd_fd_kernel<T, ORDER, 1, 1>);
        case 1: return reinterpret_cast<const void*>(&fwd_fd_kernel<T, ORDER, 2, 1>);
        case 2: return reinterpret_cast<const void*>(&fwd_fd_kernel<T, ORDER, 4, 1>);
        case 3: return reinterpret_cast<const void*>(&fwd_fd_kernel<T, ORDER, 8, 1>);
        default: return reinterpret_cast<const void*>(&fwd_fd_kernel<T, ORDER, 16, 1>);
    }
}
// One refined column a step (fd_narrow).
template <int ORDER>
const void* fd_rows_narrow(int lam) {
    switch (lam < 4 ? lam : 4) {
        case 1: return reinterpret_cast<const void*>(&fwd_fd_kernel<double, ORDER, 2, 1, false, 1>);
        case 2: return reinterpret_cast<const void*>(&fwd_fd_kernel<double, ORDER, 4, 1, false, 1>);
        case 3: return reinterpret_cast<const void*>(&fwd_fd_kernel<double, ORDER, 8, 1, false, 1>);
        case 4: return reinterpret_cast<const void*>(&fwd_fd_kernel<double, ORDER, 16, 1, false, 1>);
        default: return nullptr;
    }
}
}  // namespace

// FP64 FD calls on short paths sweep one refined column a step instead of fd_cols.  The rule counts FP64
// instructions, which bind (one per 64 cycles and quarter of an SM): a step of C columns takes k for each of
// its R C sub-cells (5 in the forward and 13 more in the adjoint, second order 7 and 19) and about o more
// (20; forward and adjoint 28 to 40, with the rows they write and read; the implicit scheme's division
// 12 and 24 on top; an inner product's d).  More columns a step spread o, but the 31 steps in which some
// lanes are not yet, or no longer, at work cost C columns each.  FP32 steps are bound by issue, where o is
// larger than the sub-cells.  Second order, lambda = 2, d = 2, one pair, a column at a time against four:
// 33 points 221 against 244 us (forward and gradients 0.67 against 0.84 ms), 65 points 735 against 589 us
// (2.10 against 2.02 ms).
bool fd_narrow(int T, int order, int lam, int64_t lx, int64_t ly, int dpad, bool tape) {
    if (T != 0 || lam == 0) return false;
    const int R = 1 << (lam < 4 ? lam : 4), C = fd_cols(R);
    const int k = order == 2 ? (tape ? 26 : 7) : (tape ? 18 : 5);
    const int o = (tape ? 16 + 6 * std::min(R, 4) : 20) + (order == 3 ? (tape ? 36 : 12) : 0) + dpad;
    const int64_t groups = (lx << lam) / R, strips = (groups + 31) / 32;
    auto cost = [&](int cols) {
        const int64_t n = (ly << lam) / cols;
        const int64_t steps = (strips - 1) * std::max<int64_t>(n, 32) + std::min<int64_t>(groups, 32) - 1 + n;
        return static_cast<double>(steps) * (R * cols * k + o);
    };
    return cost(1) < cost(C);
}

const void* fwd_interp_ptr_f32(int N) {
    if (const void* k = fwd_interp_ptr_f32_0(N)) return k; if (const void* k = fwd_interp_ptr_f32_1(N)) return k; if (const void* k = fwd_interp_ptr_f32_2(N)) return k; if (const void* k = fwd_interp_ptr_f32_3(N)) return k; if (const void* k = fwd_interp_ptr_f32_4(N)) return k;
    return nullptr;
}

const void* fwd_interp_chain_ptr_f32(int N) {
    if (const void* k = fwd_interp_chain_ptr_f32_0(N)) return k; if (const void* k = fwd_interp_chain_ptr_f32_1(N)) return k; if (const void* k = fwd_interp_chain_ptr_f32_2(N)) return k; if (const void* k = fwd_interp_chain_ptr_f32_3(N)) return k; if (const void* k = fwd_interp_chain_ptr_f32_4(N)) return k;
    return nullptr;
}

const void* fwd_interp_ptr_f64(int N) {
    if (const void* k = fwd_interp_ptr_f64_0(N)) return k; if (const void* k = fwd_interp_ptr_f64_1(N)) return k; if (const void* k = fwd_interp_ptr_f64_2(N)) return k; if (const void* k = fwd_interp_ptr_f64_3(N)) return k; if (const void* k = fwd_interp_ptr_f64_4(N)) return k;
    return nullptr;
}

const void* fwd_interp_chain_ptr_f64(int N) {
    if (const void* k = fwd_interp_chain_ptr_f64_0(N)) return k; if (const void* k = fwd_interp_chain_ptr_f64_1(N)) return k; if (const void* k = fwd_interp_chain_ptr_f64_2(N)) return k; if (const void* k = fwd_interp_chain_ptr_f64_3(N)) return k; if (const void* k = fwd_interp_chain_ptr_f64_4(N)) return k;
    return nullptr;
}

const void* fwd_interp_mt_ptr_f32(int N) {
    if (const void* k = fwd_interp_mt_ptr_f32_0(N)) return k; if (const void* k = fwd_interp_mt_ptr_f32_1(N)) return k; if (const void* k = fwd_interp_mt_ptr_f32_2(N)) return k; if (const void* k = fwd_interp_mt_ptr_f32_3(N)) return k; if (const void* k = fwd_interp_mt_ptr_f32_4(N)) return k;
    return nullptr;
}

const void* fwd_poly_kernel_ptr(int T, bool interp, int N, bool chain, bool mt, bool tape, bool mx) {
    if (chain) {
        if (tape && !interp) return T == 1 ? fwd_approx_chain_tape_ptr_f32(N) : fwd_approx_chain_tape_ptr_f64(N);
        if (T == 1) return interp ? fwd_interp_chain_ptr_f32(N) : fwd_approx_chain_ptr_f32(N);
        return interp ? fwd_interp_chain_ptr_f64(N) : fwd_approx_chain_ptr_f64(N);
    }
    if (mx) {
        if (T != 1 || interp) return nullptr;
        return tape ? fwd_approx_tape_mx_ptr_f32(N) : fwd_approx_mx_ptr_f32(N);
    }
    if (tape && !interp) {
        if (T == 1) return mt ? fwd_approx_tape_ptr_f32_mt(N) : fwd_approx_tape_ptr_f32(N);
        return mt ? nullptr : fwd_approx_tape_ptr_f64(N);
    }
    if (mt) {
        if (T != 1) return nullptr;
        return interp ? fwd_interp_mt_ptr_f32(N) : fwd_approx_mt_ptr_f32(N);
    }
    if (T == 1) return interp ? fwd_interp_ptr_f32(N) : fwd_approx_ptr_f32(N);
    return interp ? fwd_interp_ptr_f64(N) : fwd_approx_ptr_f64(N);
}

const void* fwd_fd_kernel_ptr(int T, int order, int lam, bool coop, bool tape, bool narrow, bool loop) {
    if (lam < 0 || lam > kLamMax) return nullptr;
    if (tape) return coop ? nullptr : fwd_fd_tape_ptr(T, order, lam, narrow);
    if (narrow && !coop) return order == 3 ? fd_rows_narrow<3>(lam) : order == 2 ? fd_rows_narrow<2>(lam) : fd_rows_narrow<1>(lam);
    if (order == 3) return fwd_fd_implicit_ptr(T, lam, coop, loop);
    if (coop) return fwd_fd_coop_ptr(T, order, lam, loop);
    if (T == 1) return order == 2 ? fd_rows<float, 2>(lam, loop) : fd_rows<float, 1>(lam, loop);
    return order == 2 ? fd_rows<double, 2>(lam) : fd_rows<double, 1>(lam);
}

}  // namespace sk
