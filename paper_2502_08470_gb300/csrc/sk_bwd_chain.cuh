// Tape adjoint of the polynomial schemes with a pair's strips chained over several warps
// (sk_chain.cuh): the steps, the tape and the arithmetic are those of bwd_tape_kernel, with one
// ticket per strip, taken from the top strip down.  Lane 0's left-edge adjoints go to lane 31 of the
// strip below, columns from the right edge to the left.
//
// What bounds it: as in sk_fwd_chain.cuh, the latency of a step.  The tape rows of a strip's steps
// stream into the same per-warp ring as in bwd_tape_kernel.  A step of the one-warp schedule can hold
// lanes of two strips (they overlap by 31 steps), so a warp reads whole steps and uses its own lanes,
// and writes dk/dM for its own lanes only.
#pragma once

#include "sk_bwd_poly.cuh"
#include "sk_chain.cuh"

namespace sk {

template <typename T, int N, bool INTERP>
__global__ void __launch_bounds__(kFwdWarps * 32, (bwd_tape_min_blocks<T, N, INTERP>()))
    bwd_chain_kernel(BwdParams B) {
    constexpr int NE = bwd_series_top<T, N, INTERP>();
    constexpr bool kRescale = std::is_same<T, float>::value;
    constexpr int kW = chain_words<T>(N);
    using Ends = ChainEnds<kW>;
    using Col = ChainCol<kW>;
    using V = typename Vec<T>::type;
    constexpr int W = Vec<T>::W;
    constexpr int TR = tape_row<T>(N, INTERP);
    const Launch& L = B.L;
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    constexpr int kStepBytes = fwd_tape_step_bytes<T, N, INTERP>();
    __shared__ __align__(16) uint32_t hand[kFwdWarps][Col::kWarpWords];
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char* ring = smem_raw + wib * bwd_tape_warp_bytes<T, N, INTERP>();
    uint64_t* bars = reinterpret_cast<uint64_t*>(ring + kTapeRing * kStepBytes);
    if (lane == 0) {
        for (int k = 0; k < kTapeRing; ++k) mbar_init(bars + k, 1);
        fence_mbar_init();
    }
    __syncwarp();
    uint32_t parity = 0;  // bit k: phase of slot k's barrier awaited next (warp-uniform)
    bool stuck = false;

    while (!stuck) {
        const ChainTicket tk = next_ticket(L);
        if (tk.id < 0) break;
        const int64_t item = tk.item;
        const int q = tk.strip;  // place of the strip in the pair's chain: 0 is the top strip
        const PairDesc P = decode_pair(L, item);
        if (P.lx < 0 || P.ly < 0) {
            if (lane == 0) record_error(SK_ERR_BAD_LENGTH);
            chain_finish(L, tk);
            continue;
        }
        // pairs without cells, and those the contraction skips too; every strip of a pair decides alike
        if (P.lx == 0 || P.ly == 0 || item_gbar(B, item, P) == 0.0) {
            chain_finish(L, tk);
            continue;
        }
        const int lam = L.lam;
        const int rows = static_cast<int>(P.lx << lam);
        const int cols = static_cast<int>(P.ly << lam);
        const int period = cols > 32 ? cols : 32;
        const int nstrips = (rows + 31) >> 5;
        const int s = nstrips - 1 - q;
        const int row = (s << 5) + lane;
        const int last_lane = q == 0 ? rows - 1 - (s << 5) : 31;
        const int nsteps = cols + last_lane;
        const int64_t pos0 = static_cast<int64_t>(s) * period;
        const bool in_grid = row < rows;
        const int ek = L.tape_ek[item];
        const char* tape = static_cast<const char*>(L.tape) + item * L.tape_stride + pos0 * kStepBytes;
        T* mout = reinterpret_cast<T*>(static_cast<char*>(B.mbuf) + item * B.mb_stride);
        if constexpr (std::is_same<T, float>::value) {
            if (B.gtile && q == 0) gtile_zero_padding(mout, rows, cols, B.gt_ncb);  // cells outside the grid hold zero
        }
        Ends ends;
        ends.polls = chain_polls(L, q);
        ends.stuck = false;
        ends.cols = cols;
        ends.fifo = hand[wib];
        ends.stage = hand[wib] + 2 * Col::kCols * Col::kWords;
        ends.tag_in = tk.pred;
        ends.tag_out = static_cast<uint32_t>(tk.id) + 1u;
        ends.next = ChainUnit{0ull, 0ull};
        ends.in = q > 0 ? chain_buffer(L, tk, q - 1, cols, Col::kUnits) : nullptr;
        ends.out = nullptr;

        // the corner cell (rows - 1, cols - 1) is seeded from the endpoint average, as in bwd_tape_kernel
        T gra[N + 1], gbo[N + 1];
        int gea = kZeroExp, gbe = kZeroExp;
        const bool seeded = !INTERP && q == 0 && lane == last_lane;
#pragma unroll
        for (int n = 0; n <= N; ++n) {
            gra[n] = seeded ? static_cast<T>(0.5 * cx_rfact(n)) : T(0);
            gbo[n] = T(0);
        }
        if (seeded) gea = 0;

        if (lane == 0) {
            fence_proxy_async_smem();
            for (int k = 0; k < kTapeRing && nsteps - 1 - k >= 0; ++k) {
                const int t = nsteps - 1 - k;
                const int sl = t % kTapeRing;
                mbar_arrive_expect_tx(bars + sl, kStepBytes);
                bulk_load(ring + sl * kStepBytes, tape + static_cast<int64_t>(t) * kStepBytes, kStepBytes, bars + sl);
            }
        }
        if (!chain_claim(L, tk, q + 1 < nstrips)) ends.stuck = true;
        else if (q + 1 < nstrips) ends.out = chain_buffer(L, tk, q, cols, Col::kUnits);
        ends.open();
        int stuck_step = -1;
        for (int t = nsteps - 1; t >= 0; --t) {
            const int sl = t % kTapeRing;
            if (!mbar_wait(bars + sl, (parity >> sl) & 1u)) {
                stuck = true;  // the device error word is set; drain what is in flight and stop
                stuck_step = t;
                break;
            }
            parity ^= 1u << sl;
            T fa[N + 1], fb[N + 1];  // the lane's tape row, as bwd_tape_kernel reads it
            int ef;
            T M;
            {
                const V* src = reinterpret_cast<const V*>(ring + sl * kStepBytes);
                auto put = [&](int k, T x) {
                    if constexpr (INTERP) {
                        if (k <= N) fa[k] = x;
                        else if (k <= 2 * N + 1) fb[k - N - 1] = x;
                        else if (k == 2 * N + 2) ef = exponent_from<T>(x);
                        else if (k == 2 * N + 3) M = x;
                    } else {
                        if (k < N) fa[k] = x;
                        else if (k < 2 * N) fb[k - N] = x;
                        else if (k == 2 * N) ef = exponent_from<T>(x);
                        else M = x;
                    }
                };
#pragma unroll
                for (int v = 0; v < TR / W; ++v) {
                    const V tv = src[v * 32 + lane];
                    const T* tp = reinterpret_cast<const T*>(&tv);
#pragma unroll
                    for (int w = 0; w < W; ++w) put(v * W + w, tp[w]);
                }
                if constexpr (TR % W != 0) {
                    const float2 tv = reinterpret_cast<const float2*>(ring + sl * kStepBytes + (TR / W) * 32 * 16)[lane];
                    put((TR / W) * W, tv.x);
                    put((TR / W) * W + 1, tv.y);
                }
            }
            __syncwarp();  // every lane has its row: the slot can be refilled
            if (lane == 0 && t - kTapeRing >= 0) {
                fence_proxy_async_smem();
                mbar_arrive_expect_tx(bars + sl, kStepBytes);
                bulk_load(ring + sl * kStepBytes, tape + static_cast<int64_t>(t - kTapeRing) * kStepBytes, kStepBytes,
                          bars + sl);
            }
            T gb_in[N + 1];
#pragma unroll
            for (int n = 0; n <= N; ++n) gb_in[n] = __shfl_down_sync(kFull, gbo[n], 1);
            int gbe_in = __shfl_down_sync(kFull, gbe, 1);
            const int jj = t - lane;
            const bool active = static_cast<unsigned>(jj) < static_cast<unsigned>(cols) && in_grid;
            const int c31 = cols + 30 - t;  // place of lane 31's column in the hand-off
            if (ends.in != nullptr && c31 < cols) {
                if ((c31 & (Col::kCols - 1)) == 0) ends.take(c31 / Col::kCols, 0);
                uint32_t w[Col::kWords];
                chain_words_load<kW>(ends.column(c31), w);
#pragma unroll
                for (int n = 0; n <= N; ++n) gb_in[n] = lane == 31 ? chain_value<T>(w, n) : gb_in[n];
                if constexpr (kRescale) gbe_in = lane == 31 ? static_cast<int>(w[N + 1]) : gbe_in;
                else gbe_in = lane == 31 ? 0 : gbe_in;
            }
            T mrel = T(0);
            if (active) {
                if (row == rows - 1) {  // no cell above
#pragma unroll
                    for (int n = 0; n <= N; ++n) gb_in[n] = T(0);
                    gbe_in = kZeroExp;
                }
                const bool corner = q == 0 && t == nsteps - 1;  // warp-uniform
                if (!INTERP && corner) {
#pragma unroll
                    for (int n = 0; n <= N; ++n) gb_in[n] = static_cast<T>(0.5 * cx_rfact(n));
                    gbe_in = 0;
                }
                int eg = 0;
                if (kRescale) {
                    eg = max(gea, gbe_in);
                    if (gea != eg) {
                        const T f = pow2c<T>(gea - eg);
#pragma unroll
                        for (int n = 0; n <= N; ++n) gra[n] *= f;
                    }
                    if (gbe_in != eg) {
                        const T f = pow2c<T>(gbe_in - eg);
#pragma unroll
                        for (int n = 0; n <= N; ++n) gb_in[n] *= f;
                    }
                }
                T da[N], db[N];
#pragma unroll
                for (int n = 0; n < N; ++n) { da[n] = fa[n]; db[n] = fb[n]; }
                if constexpr (INTERP) unit_scale<T, N>(fa, fb, ef);
                else unit_scale_dm<T, N>(da, db, ef);
                T e[NE + 1];
                build_exp_series<T, NE>(M, L.tau, e);
                T mbar;
                T ga_in[N + 1];
#pragma unroll
                for (int n = 0; n <= N; ++n) ga_in[n] = gra[n];
                if constexpr (INTERP) {
                    T gt[NE + 1], gr[NE + 1];
                    project_transpose<T, N, NE>(ga_in, gt);
                    project_transpose<T, N, NE>(gb_in, gr);
                    if (corner) {
#pragma unroll
                        for (int n = 0; n <= NE; ++n) {
                            gt[n] = static_cast<T>(0.5 * cx_rfact(n));
                            gr[n] = gt[n];
                        }
                        eg = 0;
                    }
                    cell_adjoint_interp<T, N, NE>(fa, fb, e, gt, gr, gra, gbo, mbar);
                } else {
                    cell_adjoint_dm<T, N>(da, db, e, ga_in, gb_in, gra, gbo, mbar);
                }
                mrel = mbar * pow2c<T>(eg + ef - ek - 2 * lam);
                gea = eg;
                if (kRescale && (t & 3) == 0) {  // keep the adjoints within [2^-64, 2^64]
                    float mag = 0.f;
#pragma unroll
                    for (int n = 0; n <= N; ++n)
                        mag = fmaxf(mag, fmaxf(fabsf(static_cast<float>(gra[n])), fabsf(static_cast<float>(gbo[n]))));
                    if (mag > 0x1p64f || (mag < 0x1p-64f && mag > 0.f)) {
                        const int sh = mag > 0x1p64f ? -64 : 64;
#pragma unroll
                        for (int n = 0; n <= N; ++n) { gra[n] *= pow2t<T>(sh); gbo[n] *= pow2t<T>(sh); }
                        gea -= sh;
                    }
                }
                gbe = gea;
                bool tiled = false;
                if constexpr (std::is_same<T, float>::value) {
                    if (B.gtile) {  // BF16 hi/lo tiles for the tensor-core contraction
                        tiled = true;
                        __nv_bfloat16 h, l;
                        split_bf16(mrel, h, l);
                        __nv_bfloat16* gt = reinterpret_cast<__nv_bfloat16*>(mout);
                        const int64_t k = gtile_index(row, jj, B.gt_ncb);
                        gt[k] = h;
                        gt[k + kGtilePlane] = l;
                    }
                }
                if (!tiled) {
                    const int64_t pos = pos0 + t;
                    mout[pos * 32 + ((lane + pos) & 31)] = mrel;  // skewed row
                }
            }
            if (ends.out != nullptr && t < cols) {  // lane 0's left edge goes to the strip below
                const int c = cols - 1 - t;
                if (lane == 0) {
                    uint32_t w[Col::kWords];
                    chain_pack<T, N>(w, gbo, gbe);
                    chain_words_store<kW>(ends.staged(c), w);
                }
                if (ends.batch_ends(c)) ends.hand_on(c);
            }
        }
        if (stuck) {  // wait (bounded) for the copies still in flight into this warp's ring
            if (lane == 0)
                for (int k = 0; k < kTapeRing && stuck_step - k >= 0; ++k) {
                    const int sl = (stuck_step - k) % kTapeRing;
                    mbar_wait(bars + sl, (parity >> sl) & 1u);
                }
        }
        __syncwarp();
        chain_finish(L, tk);
    }
}

}  // namespace sk
