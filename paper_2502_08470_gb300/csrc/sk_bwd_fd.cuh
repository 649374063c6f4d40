// Reverse-mode derivative (adjoint wavefront) of the finite-difference schemes (Definition "dyadic
// scheme", eq. (secondexplicitscheme), Remark "higherfd") from the forward tape of sweep_fd.
// The paper defines no gradient: this is the exact adjoint of the schemes' own arithmetic.
//
// A forward step of a lane (group g of R = 2^lambda node rows) covers C = fd_cols(R) columns.  Column J
// maps its state (differences v_r = k(gR+r+1, J) - k(gR+r, J), the bottom node k0 = k(gR, J)) and the
// input k1 = k(gR, J+1) from the lane below to the new differences v'_r and the top node k(gR+R, J+1):
//     k10 = k00 + v_r,  sum = k10 + k01,  d = a1 sum + m2 (sum + k00),  v'_r = v_r + d,
//     k11 = k01 + v'_r,  (k00, k01) <- (k10, k11),      starting from (k0, k1),
// with a1 = alpha - 1 and m2 = 1 - beta (m2 = 0 for first order and the implicit scheme).  The
// adjoint runs the same steps in reverse order (the reverse of the forward schedule, one warp per
// pair): from the adjoints of v' (carried from the lane's next column), of the top node (from the
// lane above, or lane 0 of the strip above through a per-warp buffer, or the endpoint seed 1) and
// of k1 as the next column's k0 (carried), it gives the adjoints of v, k0 and k1 (k1's goes down to
// the lane below) and, per sub-cell, dk/dm = abar1 da1/dm + mbar2 dm2/dm.  A coarse cell's
// 4^lambda sub-cells share m = M_ij / 4^lambda, so dk/dM_ij sums them over 4^-lambda; the lane
// covers the cell's 2^lambda rows and C of its columns in one step, the others in the steps before,
// and writes the sum, relative to 2^ek, into the contraction's dk/dM buffer for the coarse grid (the
// skewed [step][lane] rows of bwd_contract_kernel, or the tiles of the tensor-core contraction).
// FP32 carries power-of-two exponents for the adjoints as the polynomial adjoint does.
//
// The tape rows stream through a per-warp ring in shared memory, kFdRing<R> steps ahead: each
// lane copies its own 16-byte vectors of a step with cp.async (one commit group per step) and
// waits for the oldest group only when it needs that step, so the row loads no longer stall
// every step (measured: the FD1 adjoint at lambda = 0 spent most cycles waiting on its per-step
// loads, issue 30%).  A lane reads only the vectors it copied itself, so cp.async.wait_group
// orders the copy before the read without any warp-wide barrier.
#pragma once

#include <type_traits>

#include "sk_bwd_poly.cuh"
#include "sk_fwd_fd.cuh"

namespace sk {

// Steps of tape rows in flight per warp: deeper for the short rows of few node rows per lane.
template <int R>
__host__ __device__ constexpr int kFdRing() {
    return R <= 1 ? 8 : (R <= 2 ? 6 : 4);
}
// Shared-memory bytes of one warp's ring.
template <typename T, int R, int C = fd_cols(R)>
__host__ __device__ constexpr int fd_ring_warp_bytes() {
    return kFdRing<R>() * 32 * fd_tape_row<T>(R, C) * static_cast<int>(sizeof(T));
}

template <typename T, int ORDER, int R, int C = fd_cols(R)>
__global__ void __launch_bounds__(kFwdWarps * 32) bwd_fd_tape_kernel(BwdParams B) {
    constexpr bool kRescale = std::is_same<T, float>::value;
    using V = typename Vec<T>::type;
    constexpr int W = Vec<T>::W;
    constexpr int TR = fd_tape_row<T>(R, C);
    const Launch& L = B.L;
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int64_t slot = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + wib;
    char* base = static_cast<char*>(L.scratch) + slot * L.scratch_stride;
    T* rbuf = reinterpret_cast<T*>(base + B.off_rbuf);       // [col]: adjoint of lane 0's k1
    int* rexp = reinterpret_cast<int*>(base + B.off_rexp);   // [col]
    constexpr int D = kFdRing<R>();
    constexpr int kStepBytes = 32 * TR * static_cast<int>(sizeof(T));
    extern __shared__ __align__(16) unsigned char fd_smem[];
    unsigned char* ring = fd_smem + wib * fd_ring_warp_bytes<T, R, C>();  // [D][vector][lane]

    for (;;) {
        const int64_t item = next_item(L);
        if (item < 0) break;
        const PairDesc P = decode_pair(L, item);
        if (P.lx < 0 || P.ly < 0) {
            if (lane == 0) record_error(SK_ERR_BAD_LENGTH);
            continue;
        }
        if (P.lx == 0 || P.ly == 0) continue;
        if (item_gbar(B, item, P) == 0.0) continue;  // the contraction skips it too

        const int lam = L.lam;
        const int groups = static_cast<int>(P.lx);        // R = 2^lambda rows per lane: one coarse row
        const int nJ = static_cast<int>(P.ly << lam) / C; // tiles of C refined columns
        const int period = nJ > 32 ? nJ : 32;
        const int nstrips = (groups + 31) >> 5;
        const int last_lane = (groups - 1) - ((nstrips - 1) << 5);
        const int nsteps = (nstrips - 1) * period + last_lane + nJ;
        const int ek = L.tape_ek[item];
        const char* tape = static_cast<const char*>(L.tape) + item * L.tape_stride;
        // coarse-grid schedule of the dk/dM buffer: cell (32 s + r, j) at row s P' + j + r
        const int cols_c = static_cast<int>(P.ly);
        const int period_c = cols_c > 32 ? cols_c : 32;
        char* mout = static_cast<char*>(B.mbuf) + item * B.mb_stride;
        if constexpr (std::is_same<T, float>::value) {
            if (B.gtile) gtile_zero_padding(mout, groups, cols_c, B.gt_ncb);  // coarse cells outside the grid
        }

        T vbar[R];                  // adjoints of the lane's v at the tile after the current one
        T carry = T(0);             // adjoint of that tile's first bottom node (= the current one's last)
        int ge = kZeroExp;          // exponent of vbar and carry
        T k1out[C];                 // adjoints of this lane's bottom nodes J + 1 .. J + C (to lane - 1)
#pragma unroll
        for (int c = 0; c < C; ++c) k1out[c] = T(0);
        int k1e = kZeroExp;
        T mcell = T(0);             // dk/dM of the current coarse cell, relative to 2^ek
#pragma unroll
        for (int r = 0; r < R; ++r) vbar[r] = T(0);

        // this lane's vectors of steps nsteps - 1 .. nsteps - D, one commit group per step (step t
        // in slot t % D; empty groups past step 0 keep the count uniform)
        auto fetch = [&](int t) {
            if (t >= 0) {
                const V* src = reinterpret_cast<const V*>(tape + static_cast<int64_t>(t) * kStepBytes);
                V* dst = reinterpret_cast<V*>(ring + (t % D) * kStepBytes);
#pragma unroll
                for (int vv = 0; vv < TR / W; ++vv) cp_async16(dst + vv * 32 + lane, src + vv * 32 + lane);
            }
            cp_async_commit();
        };
#pragma unroll
        for (int k = 0; k < D; ++k) fetch(nsteps - 1 - k);

        int tt = nsteps - 1 - lane;
        int s = tt >= 0 ? tt / period : -1;
        int jj = tt >= 0 ? tt - s * period : -1;
        for (int step = nsteps - 1; step >= 0; --step) {
            cp_async_wait<D - 1>();  // this step's group has landed (the D - 1 after it may not)
            const V* trow = reinterpret_cast<const V*>(ring + (step % D) * kStepBytes);
            T tb[C];
#pragma unroll
            for (int c = 0; c < C; ++c) tb[c] = __shfl_down_sync(kFull, k1out[c], 1);
            int tbe = __shfl_down_sync(kFull, k1e, 1);
            const int g = (s << 5) + lane;
            const bool active = s >= 0 && jj < nJ && g < groups;
            if (active) {
                if (g == groups - 1) {            // the top group: no lane above in this pair
#pragma unroll
                    for (int c = 0; c < C; ++c) tb[c] = T(0);
                    tbe = kZeroExp;
                    if (jj == nJ - 1) {           // the endpoint k(nI, nJ): seed 1
                        tb[C - 1] = T(1);
                        tbe = 0;
                    }
                } else if (lane == 31) {          // from lane 0 of the strip above
#pragma unroll
                    for (int c = 0; c < C; ++c) tb[c] = rbuf[jj * C + c];
                    tbe = kRescale ? rexp[jj] : 0;
                }
                // the tape row of this step
                T v[R], k[C + 1], m;
                int ea = 0;
                {
#pragma unroll
                    for (int vv = 0; vv < TR / W; ++vv) {
                        const V t = trow[vv * 32 + lane];
                        const T* tp = reinterpret_cast<const T*>(&t);
#pragma unroll
                        for (int q2 = 0; q2 < W; ++q2) {
                            const int q = vv * W + q2;
                            if (q < R) v[q < R ? q : 0] = tp[q2];
                            else if (q <= R + C) k[q <= R + C ? q - R : 0] = tp[q2];
                            else if (q == R + C + 1) m = tp[q2];
                            else if (q == R + C + 2) ea = exponent_from<T>(tp[q2]);
                        }
                    }
                }
                if constexpr (kRescale && C > 1) {
                    // Far from magnitude 1, bring the tile's inputs there: their products with the
                    // adjoints (within 2^+-64) then stay in range, and a tile that the forward
                    // rescaled between its columns (|m| > kFdTileM) has the whole range to grow in.
                    const float at = fmaxf(fabsf(static_cast<float>(k[0])), fabsf(static_cast<float>(k[C])));
                    if (!(fabsf(static_cast<float>(m)) <= kFdTileM) || at > 0x1p16f || at < 0x1p-16f) {
                        float big = 0.f;
#pragma unroll
                        for (int r = 0; r < R; ++r) big = fmaxf(big, fabsf(static_cast<float>(v[r])));
#pragma unroll
                        for (int c = 0; c <= C; ++c) big = fmaxf(big, fabsf(static_cast<float>(k[c])));
                        int sh = 0;
                        if (big > 0.f) frexpf(big, &sh);
                        const T f = pow2c<T>(-sh);
#pragma unroll
                        for (int r = 0; r < R; ++r) v[r] *= f;
#pragma unroll
                        for (int c = 0; c <= C; ++c) k[c] *= f;
                        ea += sh;
                    }
                }
                if (jj == nJ - 1) {  // the lane's first reverse tile of this strip: nothing carried
#pragma unroll
                    for (int r = 0; r < R; ++r) vbar[r] = T(0);
                    carry = T(0);
                    ge = kZeroExp;
                }
                // bring the carried adjoints and the ones from above to a common exponent
                int eg = 0;
                if (kRescale) {
                    eg = max(ge, tbe);
                    if (ge != eg) {
                        const T f = pow2c<T>(ge - eg);
#pragma unroll
                        for (int r = 0; r < R; ++r) vbar[r] *= f;
                        carry *= f;
                    }
                    if (tbe != eg) {
                        const T f = pow2c<T>(tbe - eg);
#pragma unroll
                        for (int c = 0; c < C; ++c) tb[c] *= f;
                    }
                }
                // forward recompute of the tile (as sweep_fd runs it)
                T a1 = m * T(0.5);
                if constexpr (ORDER == 3) a1 = a1 / (T(1) - m * T(0.25));
                T m2 = T(0);
                if constexpr (ORDER == 2) m2 = m * m * T(1.0 / 12.0);
                T k00s[C][R], sums[C][R];
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    T k00 = k[c], k01 = k[c + 1];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const T k10 = k00 + v[r];
                        const T sum = k10 + k01;
                        T d2 = a1 * sum;
                        if constexpr (ORDER == 2) d2 = fma(m2, sum + k00, d2);
                        v[r] += d2;
                        const T k11 = k01 + v[r];
                        k00s[c][r] = k00;
                        sums[c][r] = sum;
                        k00 = k10;
                        k01 = k11;
                    }
                }
                // 2^(eg + ea - ek - 2 lambda) in two factors: the sums below can be as large as 2^111
                // where their product with it is of order 1
                const int me = eg + ea - ek - 2 * lam;
                const T mscale0 = pow2c<T>(me >> 1), mscale1 = pow2c<T>(me - (me >> 1));
#pragma unroll
                for (int c = C - 1; c >= 0; --c) {
                    // reverse of the column
                    T k01b = tb[c], k00b = T(0), a1b = T(0), m2b = T(0);
#pragma unroll
                    for (int r = R - 1; r >= 0; --r) {
                        const T k11b = k01b, k10b0 = k00b;
                        const T vpb = vbar[r] + k11b;         // v'_r: carried and through k11 = k01 + v'_r
                        T k01r = k11b;
                        T vb = vpb;                           // through v'_r = v_r + d
                        const T db = vpb;
                        T sumb = a1 * db;
                        T k00r = T(0);
                        a1b = fma(sums[c][r], db, a1b);
                        if constexpr (ORDER == 2) {
                            sumb = fma(m2, db, sumb);
                            k00r = m2 * db;
                            m2b = fma(sums[c][r] + k00s[c][r], db, m2b);
                        }
                        const T k10b = k10b0 + sumb;          // sum = k10 + k01
                        k01r += sumb;
                        k00r += k10b;                          // k10 = k00 + v_r
                        vb += k10b;
                        vbar[r] = vb;
                        k01b = k01r;
                        k00b = k00r;
                    }
                    // dk/dm of the column's R sub-cells: a1' and m2' of the scheme
                    T mb;
                    if constexpr (ORDER == 3) {
                        const T den = T(1) - m * T(0.25);
                        mb = a1b * (T(0.5) / (den * den));
                    } else {
                        mb = a1b * T(0.5);
                        if constexpr (ORDER == 2) mb = fma(m2b, m * T(1.0 / 6.0), mb);
                    }
                    mcell = fma(mb * mscale0, mscale1, mcell);
                    // k1 of this column: through this column's sub-cells and as the next column's k0
                    k1out[c] = k01b + carry;
                    carry = k00b;
                }
                ge = eg;
                // Keep the adjoints within [2^-64, 2^64]: every 4 steps for one column a step, else after
                // every tile and with what goes to the lane below (on steep paths the adjoint grows
                // from lane to lane down a strip by up to 2^31 a tile).
                if (kRescale && (C > 1 || (step & 3) == 0)) {
                    T mag = fabs(carry);
#pragma unroll
                    for (int r = 0; r < R; ++r) mag = fmax(mag, fabs(vbar[r]));
                    if constexpr (C > 1) {
#pragma unroll
                        for (int c = 0; c < C; ++c) mag = fmax(mag, fabs(k1out[c]));
                    }
                    const float fm = static_cast<float>(mag);
                    if (fm > 0x1p64f || (fm < 0x1p-64f && fm > 0.f)) {
                        const int sh = fm > 0x1p64f ? -64 : 64;
#pragma unroll
                        for (int r = 0; r < R; ++r) vbar[r] *= pow2t<T>(sh);
                        carry *= pow2t<T>(sh);
                        ge -= sh;
                        if constexpr (C > 1) {
#pragma unroll
                            for (int c = 0; c < C; ++c) k1out[c] *= pow2t<T>(sh);
                        }
                    }
                }
                k1e = C > 1 ? ge : eg;
                if (lane == 0 && s > 0) {  // hand the bottom nodes' adjoints to lane 31 of the strip below
#pragma unroll
                    for (int c = 0; c < C; ++c) rbuf[jj * C + c] = k1out[c];
                    if (kRescale) rexp[jj] = k1e;
                }
                if (((jj * C) & ((1 << lam) - 1)) == 0) {  // the coarse cell's first columns: its sum is complete
                    const int j = (jj * C) >> lam;
                    bool tiled = false;
                    if constexpr (std::is_same<T, float>::value) {
                        if (B.gtile) {
                            tiled = true;
                            __nv_bfloat16 h, l;
                            split_bf16(mcell, h, l);
                            __nv_bfloat16* gt = reinterpret_cast<__nv_bfloat16*>(mout);
                            const int64_t q = gtile_index(g, j, B.gt_ncb);
                            gt[q] = h;
                            gt[q + kGtilePlane] = l;
                        }
                    }
                    if (!tiled) {
                        const int64_t row = static_cast<int64_t>(s) * period_c + j + lane;
                        reinterpret_cast<T*>(mout)[row * 32 + ((lane + row) & 31)] = mcell;
                    }
                    mcell = T(0);
                }
            }
            fetch(step - D);  // into the slot this step's row came from
            __syncwarp();
            if (s >= 0 && --jj < 0) {  // down one strip
                jj = period - 1;
                --s;
            }
        }
        __syncwarp();
    }
}

}  // namespace sk
