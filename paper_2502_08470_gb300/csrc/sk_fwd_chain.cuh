// Forward wavefront of the polynomial schemes with a pair's strips chained over several warps
// (sk_chain.cuh): the cells, their order and their arithmetic are those of sweep_poly, so the values
// are the same bit for bit; only who computes a strip differs.
//
// What bounds it: few pairs leave few warps on the GPU, so a step's latency counts, not its issue
// slots.  Everything that a step waits for from outside the warp is therefore read ahead: the
// incoming edges a batch of columns earlier (ChainEnds), and M, in FP32, from a ring in shared
// memory that the warp fills itself, two rows of the next 16 columns a step, beside the cell's own
// chain of multiply-adds (MTile).  And what almost never happens is asked once for the warp, not
// branched on per lane: exponents that differ (`mixed`), an M beyond tau (`big`).
#pragma once

#include <type_traits>

#include "sk_chain.cuh"
#include "sk_fwd_poly.cuh"

namespace sk {

// The M of a strip, formed 16 columns at a time while the 16 before them are swept: in each step a lane
// forms one inner product, of column c0 + lane % 16 with row r or r + 8 (half-warps).  Column c, row r
// is read at step c + r, so 16 columns reach 16 + 16 + 31 steps ahead and the ring holds 64 steps.
// Element (step p, row r) sits at 32 (p mod 64) + (r + p) mod 32: a step's 32 lanes read 32 banks, and
// the two half-warps' stores (banks 2 r + c and 2 r + 16 + c) fill 32 banks as well.  A lane keeps its
// column's increment row in registers (16-byte chunks up to kRegs, the rest read from L1); the inner
// products run in row_dot's order, so M is bit for bit the value row_dot gives.
constexpr int kChainMSteps = 64;
__host__ __device__ constexpr int chain_smem_floats(int dpad) { return kChainMSteps * 32 + 32 * dpad; }  // per warp

struct MTile {
    static constexpr int kRegs = 4;
    float4 y[kRegs];
    const float4* yv;
    int c;  // this lane's column

    __device__ __forceinline__ void open(const float* __restrict__ ybase, int dpad, int lam, int cols, int c0) {
        c = c0 + (threadIdx.x & 15);
        yv = reinterpret_cast<const float4*>(ybase + static_cast<int64_t>(min(c, cols - 1) >> lam) * dpad);
#pragma unroll
        for (int k = 0; k < kRegs; ++k)
            if (4 * k < dpad) y[k] = __ldg(yv + k);
    }
    // the u-th of the 16 steps that form a tile; xs: the strip's x rows, [32][dpad]
    __device__ __forceinline__ void rows(int u, int dpad, float sub, const float* xs, float* ring) const {
        const int r = (u & 7) + (u & 8) * 2 + ((threadIdx.x & 16) >> 1);
        const float4* x = reinterpret_cast<const float4*>(xs + r * dpad);
        float acc = 0.f;
#pragma unroll
        for (int k = 0; k < kRegs; ++k)
            if (4 * k < dpad) acc = Vec<float>::dot(x[k], y[k], acc);
#pragma unroll 1
        for (int k = kRegs; 4 * k < dpad; ++k) acc = Vec<float>::dot(x[k], __ldg(yv + k), acc);
        const int p = c + r;
        ring[(p & (kChainMSteps - 1)) * 32 + ((r + p) & 31)] = acc * sub;
    }
};

// One strip (32 grid rows from 32 g) of one pair.  DMT: record the tape of output derivatives
// (approximation scheme); the interpolation scheme records its cell inputs whenever L.tape is set.
template <typename T, int N, int NE, bool INTERP, bool DMT>
__device__ __forceinline__ void sweep_strip(const Launch& L, int64_t item, const PairDesc& P, int g,
                                            ChainEnds<chain_words<T>(N)>& ends, T* xs, T* mring) {
    using Col = ChainCol<chain_words<T>(N)>;
    constexpr bool kRescale = std::is_same<T, float>::value;
    constexpr int kW = chain_words<T>(N);
    using V = typename Vec<T>::type;
    constexpr int W = Vec<T>::W;
    const int lane = threadIdx.x & 31;
    const int dpad = L.dpad;
    const int row_bytes = dpad * static_cast<int>(sizeof(T));
    const int lam = L.lam;
    const int rows = static_cast<int>(P.lx << lam);
    const int cols = static_cast<int>(P.ly << lam);
    const int period = cols > 32 ? cols : 32;  // of the one-warp schedule (tape and M layout)
    const int row = (g << 5) + lane;
    const bool last = row - lane + 32 >= rows;
    const int last_lane = last ? rows - 1 - (g << 5) : 31;
    const int nsteps = cols + last_lane;
    const bool in_grid = row < rows;
    const T sub = pow2t<T>(-2 * lam);
    const T* __restrict__ xrow = static_cast<const T*>(L.X.inc) + (P.xs + (min(row, rows - 1) >> lam)) * dpad;
    const T* __restrict__ ybase = static_cast<const T*>(L.Y.inc) + P.ys * dpad;
    constexpr bool kRing = std::is_same<T, float>::value;  // M from the warp's ring, else per cell

    T a[N + 1], bo[N + 1];
#pragma unroll
    for (int n = 0; n <= N; ++n) { a[n] = T(0); bo[n] = T(0); }
    int ea = 0, eo = 0;
    const int64_t pos0 = static_cast<int64_t>(g) * period;
    // Warp-uniform: lanes' exponents may differ (until then all are zero); an M of this step is beyond tau.
    bool mixed = false, big = !kRing;
    T M = T(0);
    MTile tile;
    if constexpr (kRing) {
        __syncwarp();  // earlier readers of xs and the ring are done
        for (int k = 0; k < dpad; k += W)
            *reinterpret_cast<V*>(xs + lane * dpad + k) = __ldg(reinterpret_cast<const V*>(xrow + k));
        __syncwarp();
        tile.open(ybase, dpad, lam, cols, 0);
#pragma unroll 1
        for (int u = 0; u < 16; ++u) tile.rows(u, dpad, sub, xs, mring);
        __syncwarp();
        M = mring[lane];
        big = __any_sync(kFull, lane == 0 && fabsf(M) > L.tau) != 0;
    }

    // k_hat = 1/2 sum_n (a_n + b_n) / n! at the last cell (interpolation: of the unprojected series)
    auto write_endpoint = [&](double twice) {
        const double v0 = 0.5 * twice;
        const double v = kRescale ? ldexp(v0, ea) : v0;
        if (!isfinite(v)) record_error(SK_ERR_NONFINITE);
        write_result(L, item, P, v);
        if (L.tape_ek != nullptr) {
            int e2 = 0;
            if (v0 != 0.0) frexp(v0, &e2);
            L.tape_ek[item] = (kRescale ? ea : 0) + e2;
        }
    };

    for (int t = 0; t < nsteps; ++t) {
        if constexpr (kRing) {
            if ((t & 15) == 0) tile.open(ybase, dpad, lam, cols, t + 16);
        }
        if (ends.in != nullptr && t < cols && (t & (Col::kCols - 1)) == 0 && ends.take(t / Col::kCols, N + 1) && kRescale)
            mixed = true;
        T b[N + 1];
#pragma unroll
        for (int n = 0; n <= N; ++n) b[n] = __shfl_up_sync(kFull, bo[n], 1);
        int eb = 0;
        if (kRescale && mixed) eb = __shfl_up_sync(kFull, eo, 1);
        const int jj = t - lane;
        const bool active = static_cast<unsigned>(jj) < static_cast<unsigned>(cols) && in_grid;
        if (ends.in != nullptr) {  // lane 0 takes the edge that the strip before handed on
            uint32_t w[Col::kWords];
            chain_words_load<kW>(ends.column(t), w);
#pragma unroll
            for (int n = 0; n <= N; ++n) b[n] = lane == 0 ? chain_value<T>(w, n) : b[n];
            if constexpr (kRescale) eb = lane == 0 ? static_cast<int>(w[N + 1]) : eb;
        } else {  // q^{0,j} = e_0 (left boundary k(0, .) = 1)
#pragma unroll
            for (int n = 0; n <= N; ++n) b[n] = lane == 0 ? (n == 0 ? T(1) : T(0)) : b[n];
            eb = lane == 0 ? 0 : eb;
        }
        if (t < 32) {  // p^{i,0} = e_0 (bottom boundary k(., 0) = 1)
#pragma unroll
            for (int n = 0; n <= N; ++n) a[n] = jj == 0 ? (n == 0 ? T(1) : T(0)) : a[n];
        }
        if (kRescale && mixed && active && ea != eb) {  // bring both inputs to the larger exponent
            if (ea > eb) {
                const T f = (eb - ea < -126) ? T(0) : pow2t<T>(eb - ea);
#pragma unroll
                for (int n = 0; n <= N; ++n) b[n] *= f;
            } else {
                const T f = (ea - eb < -126) ? T(0) : pow2t<T>(ea - eb);
#pragma unroll
                for (int n = 0; n <= N; ++n) a[n] *= f;
                ea = eb;
            }
        }
        T Mnext = T(0);
        if constexpr (kRing) {
            M = active ? M : 0.f;
            Mnext = mring[((t + 1) & (kChainMSteps - 1)) * 32 + ((lane + t + 1) & 31)];
        } else {
            const int jc = min(max(jj, 0), cols - 1);
            M = row_dot<T>(xrow, row_at(ybase, jc >> lam, row_bytes), L.nvec) * sub;
        }
        if constexpr (INTERP) {
            if (L.tape != nullptr && active) {  // the cell's inputs (layout as in sweep_poly)
                constexpr int TR = tape_row<T>(N, true);
                constexpr int kStepBytes = 32 * TR * static_cast<int>(sizeof(T));
                V* dst = reinterpret_cast<V*>(static_cast<char*>(L.tape) + item * L.tape_stride + (pos0 + t) * kStepBytes);
#pragma unroll
                for (int v = 0; v < TR / W; ++v) {
                    V tv;
                    T* tp = reinterpret_cast<T*>(&tv);
#pragma unroll
                    for (int q2 = 0; q2 < W; ++q2) {
                        const int q = v * W + q2;
                        tp[q2] = q <= N ? a[q] : (q <= 2 * N + 1 ? b[q - N - 1] : T(0));
                        if (q == 2 * N + 2) tp[q2] = exponent_as<T>(ea);
                        if (q == 2 * N + 3) tp[q2] = M;
                    }
                    __stcs(dst + v * 32 + lane, tv);
                }
            }
        }
        T e[NE + 1];
        build_small_exp_series<T, NE>(M, e);
        if (big) {
            // The compiler forms the short FP64 series of orders 2 and 3 in every step and selects; a value that
            // exists only here keeps it in the branch (1326 pairs of 257 points, order 3: 1.41 -> 0.79 ms, order
            // 2: 0.90 -> 0.73).  Longer series stay in it by themselves, and ran 2% slower this way.
            T m = M;
            if constexpr (std::is_same<T, float>::value && NE <= 3) asm volatile("" : "+f"(m));
            build_exp_series<T, NE>(m, L.tau, e);
        }
        const bool at_end = active && row == rows - 1 && jj == cols - 1;
        if constexpr (std::is_same<T, float>::value && !INTERP) {  // (pairs lose on the longer interpolation series)
            float2 c[NE + 1];
            if constexpr (DMT) {
                float2 dm[N];
                cell_pairs_dm<N>(a, b, e, c, dm);
                float da[N], db[N];
#pragma unroll
                for (int n = 0; n < N; ++n) { da[n] = dm[n].x; db[n] = dm[n].y; }
                if (active)  // other lanes' rows of this step belong to the strips beside this one
                    store_dm_row<T, N>(static_cast<char*>(L.tape) + item * L.tape_stride, static_cast<int>(pos0) + t, lane,
                                       da, db, ea, M);
            } else {
                cell_pairs<N>(a, b, e, c);
            }
#pragma unroll
            for (int n = 0; n <= N; ++n) { a[n] = c[n].x; bo[n] = c[n].y; }
        } else {
            T ct[NE + 1], cr[NE + 1];
            if constexpr (DMT) {
                T da[N], db[N];
                cell_series_dm<T, N>(a, b, e, ct, cr, da, db);
                if (active)
                    store_dm_row<T, N>(static_cast<char*>(L.tape) + item * L.tape_stride, static_cast<int>(pos0) + t, lane,
                                       da, db, ea, M);
            } else {
                cell_series<T, N, NE, INTERP>(a, b, e, ct, cr);
            }
            if (INTERP && at_end) write_endpoint(series_at_one<T, NE>(ct) + series_at_one<T, NE>(cr));
            project_both<T, N, NE, INTERP>(ct, cr, a, bo);
        }
        if (kRescale && (t & 3) == 0) {
            const float mag = fmaxf(fabsf(static_cast<float>(a[0])), fabsf(static_cast<float>(bo[0])));
            if (__any_sync(kFull, active && (mag > 0x1p64f || mag < 0x1p-64f))) {
                if (!active) {
                } else if (mag > 0x1p64f) {
#pragma unroll
                    for (int n = 0; n <= N; ++n) { a[n] *= pow2t<T>(-64); bo[n] *= pow2t<T>(-64); }
                    ea += 64;
                } else if (mag < 0x1p-64f) {
                    float full = 0.f;
#pragma unroll
                    for (int n = 0; n <= N; ++n)
                        full = fmaxf(full, fmaxf(fabsf(static_cast<float>(a[n])), fabsf(static_cast<float>(bo[n]))));
                    if (full < 0x1p-64f && full > 0.f) {
#pragma unroll
                        for (int n = 0; n <= N; ++n) { a[n] *= pow2t<T>(64); bo[n] *= pow2t<T>(64); }
                        ea -= 64;
                    }
                }
                mixed = true;
            }
        }
        eo = ea;
        if (ends.out != nullptr && t >= 31) {  // lane 31's right edge goes to the next strip
            const int c = t - 31;
            if (lane == 31) {
                uint32_t w[Col::kWords];
                chain_pack<T, N>(w, bo, eo);
                chain_words_store<kW>(ends.staged(c), w);
            }
            if (ends.batch_ends(c)) ends.hand_on(c);
        }
        if constexpr (kRing) {
            big = __any_sync(kFull, static_cast<unsigned>(jj + 1) < static_cast<unsigned>(cols) && fabsf(Mnext) > L.tau) != 0;
            M = Mnext;
            tile.rows(t & 15, dpad, sub, xs, mring);
            __syncwarp();
        }
    }
    if constexpr (!INTERP) {  // the last cell was the last step of lane last_lane
        if (last && lane == last_lane) write_endpoint(series_at_one<T, N>(a) + series_at_one<T, N>(bo));
    }
}

// Persistent: blocks of kFwdWarps independent warps, a ticket at a time.  Dynamic shared memory (FP32):
// each warp's ring of M and its strip's x rows (chain_smem_floats).
// Four blocks (16 warps, 128 registers): a warp's own latency counts for more here than the number of
// warps.  Five blocks measured slower on one pair of 4096 x 4096 cells (5.51 against 4.88 ms) and on 48
// (10.8 against 9.65 ms), three the same.
template <typename T, int N, int NE>
constexpr int fwd_chain_min_blocks() {
    constexpr int b = fwd_poly_min_blocks<T, N, NE, false>();
    return b > 4 ? 4 : b;
}

template <typename T, int N, int NE, bool INTERP, bool DMT = false>
__global__ void __launch_bounds__(kFwdWarps * 32, (fwd_chain_min_blocks<T, N, NE>()))
    fwd_chain_kernel(Launch L, int64_t buf_cols) {
    using Ends = ChainEnds<chain_words<T>(N)>;
    const int wib = threadIdx.x >> 5;
    __shared__ __align__(16) uint32_t hand[kFwdWarps][Ends::Col::kWarpWords];
    extern __shared__ __align__(128) unsigned char fwd_smem[];
    T* mring = reinterpret_cast<T*>(fwd_smem) + wib * chain_smem_floats(L.dpad);
    T* xs = mring + kChainMSteps * 32;
    (void)buf_cols;
    for (;;) {
        const ChainTicket tk = next_ticket(L);
        if (tk.id < 0) break;
        const int g = tk.strip;
        const PairDesc P = decode_pair(L, tk.item);
        if (trivial_pair(L, tk.item, P)) {  // one ticket, nothing handed on
            chain_finish(L, tk);
            continue;
        }
        const int nstrips = static_cast<int>(((P.lx << L.lam) + 31) >> 5);
        Ends ends;
        ends.polls = chain_polls(L, g);
        ends.stuck = false;
        ends.cols = static_cast<int>(P.ly << L.lam);
        ends.fifo = hand[wib];
        ends.stage = hand[wib] + 2 * Ends::Col::kCols * Ends::Col::kWords;
        ends.tag_in = tk.pred;
        ends.tag_out = static_cast<uint32_t>(tk.id) + 1u;
        ends.next = ChainUnit{0ull, 0ull};
        ends.in = g > 0 ? chain_buffer(L, tk, g - 1, ends.cols, Ends::Col::kUnits) : nullptr;
        ends.out = nullptr;
        if (!chain_claim(L, tk, g + 1 < nstrips)) ends.stuck = true;
        else if (g + 1 < nstrips) ends.out = chain_buffer(L, tk, g, ends.cols, Ends::Col::kUnits);
        ends.open();
        sweep_strip<T, N, NE, INTERP, DMT>(L, tk.item, P, g, ends, xs, mring);
        __syncwarp();  // every lane is done with the incoming buffer
        chain_finish(L, tk);
    }
}

}  // namespace sk
