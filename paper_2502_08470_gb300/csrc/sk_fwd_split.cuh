// Forward wavefront in FP64 of a few short pairs (one strip, at most 32 grid rows): four warps share the
// cells of one pair, each computing some of every cell's outputs.
//
// What bounds it: a warp issues one FP64 instruction every 64 cycles, whatever number of its lanes is
// active, because each quarter of an SM has its own share of the FP64 units; four warps on the four
// quarters together issue four every 76 cycles (measured, independent multiply-adds).  One warp per
// pair therefore runs a 33-point pair at a quarter of one SM's rate while the rest of the GPU idles:
// about 75 instructions a step, 63 steps, 150 us.  Splitting lanes would not help; splitting the
// outputs c_n of a cell's two edges does: each warp forms M and the series e_m itself, then its outputs,
// and all of them exchange the edges through shared memory once a step (twice with the interpolation
// scheme's projection).  A call with one 33-point pair, order 4: 174 -> 84 us.  The sums are cell_series's, term by term in its order, so the values are the
// same bit for bit.
#pragma once

#include "sk_fwd_poly.cuh"

namespace sk {

constexpr int kSplitWarps = 4;

// Which warp computes output (edge, n), q = 2 n + edge: the costliest first, each to the warp with
// the least so far.  Cost of c_n: N multiply-adds of the coupling, the convolution's terms, the scaling.
template <int N, int NE>
struct SplitPlan {
    int owner[2 * (NE + 1)] = {};
    constexpr SplitPlan() {
        int load[kSplitWarps] = {};
        bool taken[2 * (NE + 1)] = {};
        for (int i = 0; i < 2 * (NE + 1); ++i) {
            int best = -1, cost = -1;
            for (int q = 0; q < 2 * (NE + 1); ++q) {
                const int n = q / 2;
                const int c = N + (n == 0 ? 0 : (n <= N ? n : N + 1));
                if (!taken[q] && c > cost) {
                    best = q;
                    cost = c;
                }
            }
            int w = 0;
            for (int k = 1; k < kSplitWarps; ++k)
                if (load[k] < load[w]) w = k;
            taken[best] = true;
            owner[best] = w;
            load[w] += cost;
        }
    }
};

// Barrier of the block's four warps, which run different code (one instantiation of the sweep each).
__device__ __forceinline__ void split_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(kSplitWarps * 32) : "memory"); }

// Output n of one edge: x is the edge the convolution runs over (c_0 = corner), y the other one.
template <int N, int NE, int n>
__device__ __forceinline__ double split_output(const double (&x)[N + 1], const double (&y)[N + 1], double corner,
                                               const double (&e)[NE + 1]) {
    double t = corner;
#pragma unroll
    for (int k = 1; k <= N; ++k) t = fma(y[k], Tab<double>::hank(n, k), t);
    if constexpr (n == 0) {
        return t;
    } else {
        double v;
        if constexpr (n <= N) v = x[n];
        else v = x[N] * e[n - N];
#pragma unroll
        for (int k = (n <= N ? n : N) - 1; k >= 1; --k) v = fma(x[k], e[n - k], v);
        return fma(e[n], t, v);
    }
}

template <int N, int NE, bool INTERP, int W, int n = 0>
__device__ __forceinline__ void split_outputs(const double (&a)[N + 1], const double (&b)[N + 1], const double (&e)[NE + 1],
                                              double* c) {
    constexpr SplitPlan<N, NE> plan{};
    const int lane = threadIdx.x & 31;
    if constexpr (plan.owner[2 * n] == W) c[(2 * n) * 32 + lane] = split_output<N, NE, n>(a, b, a[0], e);
    if constexpr (plan.owner[2 * n + 1] == W)
        c[(2 * n + 1) * 32 + lane] = split_output<N, NE, n>(b, a, INTERP ? a[0] : b[0], e);
    if constexpr (n < NE) split_outputs<N, NE, INTERP, W, n + 1>(a, b, e, c);
}

// Shared memory, in doubles: a cell's outputs [2 (NE + 1)][32], twice for the approximation scheme
// (written and read in turn), once plus the projected edges [2 (N + 1)][32] for the interpolation scheme.
template <int N, int NE, bool INTERP>
__host__ __device__ constexpr int split_smem_doubles() {
    return INTERP ? (2 * (NE + 1) + 2 * (N + 1)) * 32 : 2 * 2 * (NE + 1) * 32;
}

template <int N, int NE, bool INTERP, int W>
__device__ __forceinline__ void sweep_split(const Launch& L, int64_t item, const PairDesc& P, double* sm) {
    const int lane = threadIdx.x & 31;
    const int dpad = L.dpad, lam = L.lam;
    const int rows = static_cast<int>(P.lx << lam);
    const int cols = static_cast<int>(P.ly << lam);
    const int nsteps = rows - 1 + cols;
    const double sub = pow2d(-2 * lam);
    const double* xrow = static_cast<const double*>(L.X.inc) + (P.xs + (min(lane, rows - 1) >> lam)) * dpad;
    const double* ybase = static_cast<const double*>(L.Y.inc) + P.ys * dpad;
    constexpr int kOut = 2 * (NE + 1) * 32;
    for (int t = 0; t < nsteps; ++t) {
        const int jj = t - lane;
        // the edges the lane's cell starts from: (a, b) at 2 n + edge of the step before, b from one lane down
        const double* from = INTERP ? sm + kOut : sm + ((t + 1) & 1) * kOut;
        double a[N + 1], b[N + 1];
#pragma unroll
        for (int n = 0; n <= N; ++n) {
            const double unit = n == 0 ? 1.0 : 0.0;
            a[n] = jj <= 0 ? unit : from[(2 * n) * 32 + lane];                  // bottom boundary k(., 0) = 1
            b[n] = lane == 0 || t == 0 ? unit : from[(2 * n + 1) * 32 + lane - 1];  // left boundary k(0, .) = 1
        }
        const int jc = min(max(jj, 0), cols - 1);
        const double M = row_dot<double>(xrow, ybase + static_cast<int64_t>(jc >> lam) * dpad, L.nvec) * sub;
        double e[NE + 1];
        build_exp_series<double, NE>(M, L.tau, e);
        double* c = INTERP ? sm : sm + (t & 1) * kOut;
        split_outputs<N, NE, INTERP, W>(a, b, e, c);
        split_barrier();
        if (t == nsteps - 1) break;
        if constexpr (INTERP) {  // project: row n of both edges to warp n mod 4
            double* to = sm + kOut;
#pragma unroll
            for (int n = W; n <= N; n += kSplitWarps) {
                double vt = c[(2 * n) * 32 + lane], vr = c[(2 * n + 1) * 32 + lane];
#pragma unroll
                for (int j = N + 1; j <= NE; ++j) {
                    vt = fma(Tab<double>::proj(N, n, j - N - 1), c[(2 * j) * 32 + lane], vt);
                    vr = fma(Tab<double>::proj(N, n, j - N - 1), c[(2 * j + 1) * 32 + lane], vr);
                }
                to[(2 * n) * 32 + lane] = vt;
                to[(2 * n + 1) * 32 + lane] = vr;
            }
            split_barrier();
        }
    }
    if (W == 0 && lane == rows - 1) {  // the last cell: k_hat = 1/2 sum_n (a_n + b_n) / n!
        const double* c = INTERP ? sm : sm + ((nsteps - 1) & 1) * kOut;
        double ct[NE + 1], cr[NE + 1];
#pragma unroll
        for (int n = 0; n <= NE; ++n) {
            ct[n] = c[(2 * n) * 32 + lane];
            cr[n] = c[(2 * n + 1) * 32 + lane];
        }
        const double v = 0.5 * (series_at_one<double, NE>(ct) + series_at_one<double, NE>(cr));
        if (!isfinite(v)) record_error(SK_ERR_NONFINITE);
        write_result(L, item, P, v);
    }
}

// One block of four warps per pair, pairs from the queue.
template <int N, int NE, bool INTERP>
__global__ void __launch_bounds__(kSplitWarps * 32) fwd_split_kernel(Launch L, int64_t buf_cols) {
    __shared__ double sm[split_smem_doubles<N, NE, INTERP>()];
    __shared__ long long s_item;
    (void)buf_cols;
    for (;;) {
        if (threadIdx.x == 0) s_item = pop_item(L);
        __syncthreads();
        const int64_t item = s_item;
        __syncthreads();  // every warp has the item, and is done with the pair before
        if (item < 0) return;
        const PairDesc P = decode_pair(L, item);
        if (P.lx <= 0 || P.ly <= 0) {
            if (threadIdx.x < 32) trivial_pair(L, item, P);
            continue;
        }
        switch (threadIdx.x >> 5) {
            case 0: sweep_split<N, NE, INTERP, 0>(L, item, P, sm); break;
            case 1: sweep_split<N, NE, INTERP, 1>(L, item, P, sm); break;
            case 2: sweep_split<N, NE, INTERP, 2>(L, item, P, sm); break;
            default: sweep_split<N, NE, INTERP, 3>(L, item, P, sm); break;
        }
    }
}

}  // namespace sk
