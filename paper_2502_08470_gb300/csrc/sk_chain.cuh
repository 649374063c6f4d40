// Strip chain: the hand-off between the warps that sweep one pair together.
//
// A pair of S strips (32 grid rows each) swept by one warp is a serial chain of about S x cols
// steps.  When a batch has too few pairs to fill the GPU that way, or a few long ones among many,
// each strip is a work item of its own (a "ticket"): a warp takes (pair, strip) tickets from a queue
// and sweeps one strip at a time, reading the edges that the strip before it hands on while that
// strip is still being swept.
//
// Order of the tickets: by the steps that remain from the strip to the end of its pair,
// (S - s) kChainLag + cols, most first, in buckets of kChainLag.  A pair's strips thus lie in different
// buckets, each after the one it depends on, and are taken about when that one is far enough ahead; a
// warp rarely holds a strip that cannot start yet.  (A model of the uneven batch, 4096 pairs of
// 64 .. 4096 points, keeps 4256 warps busy 0.94 of the time; taking a pair's strips one after another
// 0.37.)  Every wait points at a ticket that was taken earlier, so it has finished or a running warp
// holds it, whatever the grid size and however the blocks are scheduled: no launch has to be
// co-resident.
//
// The hand-off goes through global memory as tagged words: a 16-byte unit holds two 32-bit payload
// words, each beside the producer's ticket number + 1, written and read as 64-bit relaxed accesses
// (which cannot tear), so a word that shows the right tag is itself the data: no fence and no flag
// to order.  (The ring of blocks that this replaced published progress with release stores and read
// it with acquires, 3.0 us a step.)  The buffers are cleared before a launch, so no tag of an earlier
// call is taken for one of this call's.  The consumer reads kCols columns at a time, one batch ahead
// of their use, into a small buffer in shared memory; the producer gathers as many there before it
// writes them.
//
// Buffers.  A pair has a buffer for each strip that hands on, or ch_ring of them used in turn
// (strip s then waits until strip s - ch_ring + 1 is done, ch_done[pair]).  When not all pairs' fit
// the workspace, pairs are put into groups, largest first, each of which fits half of it; a group's
// tickets come after the group before's, and wait until the group that used their half is done
// (ch_gdone).
//
// Bounds of the waits.  A wait for a column ends after a number of polls, since the strip before it is
// at work (its own wait for buffers is over, chain_claim).  A wait for buffers can last as long as a
// whole group's sweep, or several groups' in turn; it goes on as long as strips of the launch finish
// (ch_finished) and ends after a stretch without any, as long as one strip's sweep may take
// (chain_claim_polls).  Of the tickets not done, the first in the order waits for nothing that is not
// done, so one finishes in every such stretch.  A ticket whose wait for buffers ran out hands nothing on:
// the memory still belongs to others.
#pragma once

#include "sk_common.cuh"

namespace sk {

// Layout of one column of a hand-off: W payload words, two to a 16-byte unit.
template <int W>
struct ChainCol {
    static constexpr int kUnits = (W + 1) / 2;
    static_assert(kUnits <= 32, "a column's units are read by one warp");
    // Columns of a batch: as many as a warp's 32 units hold, a power of two up to 8.  More would
    // cost fewer instructions a column, but every strip starts that much later than the one before.
    static constexpr int kCols = 32 / kUnits >= 8 ? 8 : (32 / kUnits >= 4 ? 4 : (32 / kUnits >= 2 ? 2 : 1));
    static constexpr int kWords = 2 * kUnits;                    // words of a column, padded
    static constexpr int kWarpWords = 3 * kCols * kWords;        // two incoming batches, one outgoing
};

struct alignas(16) ChainUnit {
    unsigned long long a, b;  // payload in the low half, tag in the high half
};

__device__ __forceinline__ ChainUnit chain_load(const ChainUnit* p) {
    ChainUnit u;
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(u.a), "=l"(u.b) : "l"(p) : "memory");
    return u;
}
__device__ __forceinline__ void chain_store(ChainUnit* p, uint32_t w0, uint32_t w1, uint32_t tag) {
    const unsigned long long t = static_cast<unsigned long long>(tag) << 32;
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(t | w0), "l"(t | w1) : "memory");
}

// A column's words between shared memory and registers, in the widest accesses its size allows.
template <int W>
__device__ __forceinline__ void chain_words_load(const uint32_t* p, uint32_t (&w)[ChainCol<W>::kWords]) {
    constexpr int U = ChainCol<W>::kUnits;
    if constexpr (U % 2 == 0) {
#pragma unroll
        for (int k = 0; k < U / 2; ++k) {
            const uint4 v = reinterpret_cast<const uint4*>(p)[k];
            w[4 * k] = v.x;
            w[4 * k + 1] = v.y;
            w[4 * k + 2] = v.z;
            w[4 * k + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const uint2 v = reinterpret_cast<const uint2*>(p)[k];
            w[2 * k] = v.x;
            w[2 * k + 1] = v.y;
        }
    }
}
template <int W>
__device__ __forceinline__ void chain_words_store(uint32_t* p, const uint32_t (&w)[ChainCol<W>::kWords]) {
    constexpr int U = ChainCol<W>::kUnits;
    if constexpr (U % 2 == 0) {
#pragma unroll
        for (int k = 0; k < U / 2; ++k)
            reinterpret_cast<uint4*>(p)[k] = make_uint4(w[4 * k], w[4 * k + 1], w[4 * k + 2], w[4 * k + 3]);
    } else {
#pragma unroll
        for (int k = 0; k < U; ++k) reinterpret_cast<uint2*>(p)[k] = make_uint2(w[2 * k], w[2 * k + 1]);
    }
}
// Value n of a column's words, and the words of N + 1 values with an exponent (FP32).
template <typename T, int K>
__device__ __forceinline__ T chain_value(const uint32_t (&w)[K], int n) {
    if constexpr (sizeof(T) == 4) return __uint_as_float(w[n]);
    else return __hiloint2double(static_cast<int>(w[2 * n + 1]), static_cast<int>(w[2 * n]));
}
template <typename T, int N, int K>
__device__ __forceinline__ void chain_pack(uint32_t (&w)[K], const T (&v)[N + 1], int exponent) {
#pragma unroll
    for (int n = 0; n <= N; ++n) {
        if constexpr (sizeof(T) == 4) {
            w[n] = __float_as_uint(v[n]);
        } else {
            w[2 * n] = static_cast<uint32_t>(__double2loint(v[n]));
            w[2 * n + 1] = static_cast<uint32_t>(__double2hiint(v[n]));
        }
    }
    if constexpr (sizeof(T) == 4) w[N + 1] = static_cast<uint32_t>(exponent);
#pragma unroll
    for (int k = (N + 1) * static_cast<int>(sizeof(T) / 4) + (sizeof(T) == 4 ? 1 : 0); k < K; ++k) w[k] = 0u;
}

// The two ends of a ticket's hand-off, for one warp.  Columns are numbered in the order they are
// handed on.
template <int W>
struct ChainEnds {
    using Col = ChainCol<W>;
    static constexpr int kLive = Col::kCols * Col::kUnits;  // lanes that carry a unit of a batch
    const ChainUnit* in;   // the producer's buffer (NULL: no strip before this one)
    ChainUnit* out;        // this ticket's buffer (NULL: no strip after this one)
    uint32_t tag_in, tag_out;
    uint32_t* fifo;        // shared memory: [2][kCols][kWords]
    uint32_t* stage;       // shared memory: [kCols][kWords]
    int cols;
    uint32_t polls;        // polls a wait makes before it gives up
    bool stuck;
    ChainUnit next;        // the next batch's units, as last read

    __device__ __forceinline__ bool unit_ready(int batch) const {
        const int lane = threadIdx.x & 31;
        const int col = batch * Col::kCols + lane / Col::kUnits;
        if (lane >= kLive || col >= cols) return true;
        return static_cast<uint32_t>(next.a >> 32) == tag_in && static_cast<uint32_t>(next.b >> 32) == tag_in;
    }
    __device__ __forceinline__ void read_ahead(int batch) {
        const int lane = threadIdx.x & 31;
        const int col = batch * Col::kCols + lane / Col::kUnits;
        if (lane < kLive && col < cols) next = chain_load(in + static_cast<int64_t>(batch) * kLive + lane);
    }
    __device__ __forceinline__ void open() {
        if (in != nullptr) read_ahead(0);
    }
    // Batch `batch` (whose units were read ahead) into shared memory; waits, a bounded number of
    // polls, until the producer has written it.  Returns whether payload word `word` of any of its
    // columns is nonzero.  Warp-uniform.
    __device__ __forceinline__ bool take(int batch, int word) {
        const int lane = threadIdx.x & 31;
        uint32_t left = polls;
        while (!stuck && !__all_sync(kFull, unit_ready(batch))) {
            if (left-- == 0) {
                if (lane == 0) record_error(SK_ERR_DEVICE_TIMEOUT);
                stuck = true;
                break;
            }
            __nanosleep(32);
            read_ahead(batch);
        }
        const uint2 w = make_uint2(static_cast<uint32_t>(next.a), static_cast<uint32_t>(next.b));
        if (lane < kLive) *reinterpret_cast<uint2*>(fifo + (batch & 1) * Col::kCols * Col::kWords + 2 * lane) = w;
        const bool mine = lane < kLive && lane % Col::kUnits == word / 2 && batch * Col::kCols + lane / Col::kUnits < cols &&
                          (word % 2 ? w.y : w.x) != 0u;
        const bool any = __any_sync(kFull, mine) != 0;
        __syncwarp();
        read_ahead(batch + 1);
        return any;
    }
    __device__ __forceinline__ const uint32_t* column(int c) const {
        return fifo + (c & (2 * Col::kCols - 1)) * Col::kWords;
    }
    // Where the lane that produces column c puts its words, and the write of a whole batch (after
    // column c, the last of its batch or of the strip).  Warp-uniform.
    __device__ __forceinline__ uint32_t* staged(int c) const { return stage + (c & (Col::kCols - 1)) * Col::kWords; }
    __device__ __forceinline__ bool batch_ends(int c) const { return (c & (Col::kCols - 1)) == Col::kCols - 1 || c == cols - 1; }
    __device__ __forceinline__ void hand_on(int c) {
        const int lane = threadIdx.x & 31;
        __syncwarp();
        const int batch = c / Col::kCols;
        const int col = batch * Col::kCols + lane / Col::kUnits;
        if (lane < kLive && col < cols) {
            const uint2 w = *reinterpret_cast<const uint2*>(stage + 2 * lane);
            chain_store(out + static_cast<int64_t>(batch) * kLive + lane, w.x, w.y, tag_out);
        }
        __syncwarp();
    }
};

// Words of a forward or reverse hand-off column: N + 1 values, and an exponent in FP32.
template <typename T>
__host__ __device__ constexpr int chain_words(int N) {
    return (N + 1) * (static_cast<int>(sizeof(T)) / 4) + (sizeof(T) == 4 ? 1 : 0);
}
// 16-byte units that a slot holds per column (a batch's units are contiguous, so a column takes
// kLive / kCols = kUnits of them), rounded up to whole batches by the host.
template <typename T>
__host__ __device__ constexpr int chain_units(int N) {
    return (chain_words<T>(N) + 1) / 2;
}

// Steps by which a strip starts after the one below it: 31 for the wavefront, two batches of columns
// and the latency of the hand-off.
constexpr int kChainLag = 50;

struct ChainTicket {
    int64_t id;      // place in the order, -1 when none is left
    int64_t item;
    int strip;       // 0 = the strip that starts the chain
    uint32_t pred;   // the ticket of the strip before, + 1
    int group;
};

// Takes the next ticket (lane 0 pops it, every lane receives it).
__device__ __forceinline__ ChainTicket next_ticket(const Launch& L) {
    unsigned int k = 0;
    int4 t = make_int4(0, 0, 0, 0);
    if ((threadIdx.x & 31) == 0) {
        k = atomicAdd(L.queue, 1u);
        if (k < *L.ch_total) t = L.ch_tickets[k];
        else k = 0xffffffffu;
    }
    k = __shfl_sync(kFull, k, 0);
    ChainTicket c;
    c.id = k == 0xffffffffu ? -1 : static_cast<int64_t>(k);
    c.item = __shfl_sync(kFull, t.x, 0);
    c.strip = __shfl_sync(kFull, t.y, 0);
    c.pred = static_cast<uint32_t>(__shfl_sync(kFull, t.z, 0));
    c.group = __shfl_sync(kFull, t.w, 0);
    return c;
}

// The buffer that strip `strip` of the item writes (the next one reads).
__device__ __forceinline__ ChainUnit* chain_buffer(const Launch& L, const ChainTicket& c, int strip, int cols, int units) {
    const int64_t stride = static_cast<int64_t>((cols + 7) / 8 * 8) * units;
    return L.ch_hand + L.ch_base[c.item] + (strip % L.ch_ring) * stride;
}

// A wait for finished strips (*p >= need): over when no strip of the launch has finished during `polls`
// polls; false (and the device error word set) then.
__device__ __forceinline__ bool chain_wait(const Launch& L, const int* p, int need, uint32_t polls) {
    int seen = acquire_gpu(L.ch_finished);
    for (;;) {
        for (uint32_t it = 0; it < polls; ++it) {
            if (acquire_gpu(p) >= need) return true;
            __nanosleep(64);
        }
        const int now = acquire_gpu(L.ch_finished);
        if (now == seen) break;
        seen = now;
    }
    record_error(SK_ERR_DEVICE_TIMEOUT);
    return false;
}

// Polls of one stretch of such a wait.  A poll takes 0.5 us or more, so the default limit gives each of
// kChainWaitSteps steps of a sweep 2 ms, where the slowest (FP64 interpolation of the highest order, four
// warps to a quarter of an SM) takes about 0.2 ms.
constexpr int kChainWaitSteps = 256;
__device__ __forceinline__ uint32_t chain_claim_polls(const Launch& L) {
    const unsigned long long p = static_cast<unsigned long long>(wait_polls(L)) * (1 + (L.ch_cols + 31) / kChainWaitSteps);
    return p > 0xfffffff0ull ? 0xfffffff0u : static_cast<uint32_t>(p);
}

// Waits until the buffer that the ticket writes is free and the strip before it has passed the same wait
// (so that a wait for that strip's columns is a wait for a strip at work).  hands_on: a strip comes after
// this one.  False when the wait ran out: the ticket must not write then.  Warp-uniform.
__device__ __forceinline__ bool chain_claim(const Launch& L, const ChainTicket& c, bool hands_on) {
    bool ok = true;
    if ((threadIdx.x & 31) == 0) {
        const uint32_t polls = chain_claim_polls(L);
        if (c.group >= 2)
            ok = chain_wait(L, reinterpret_cast<const int*>(L.ch_gdone) + c.group - 2, static_cast<int>(L.ch_gsize[c.group - 2]), polls);
        const int writer = hands_on ? c.strip : c.strip - 1;
        if (ok && writer >= L.ch_ring) ok = chain_wait(L, L.ch_done + c.item, writer - L.ch_ring + 2, polls);
    }
    return __shfl_sync(kFull, ok ? 1 : 0, 0) != 0;
}

// Marks the ticket done.  Call after a warp barrier that follows its last read of the buffer before it.
__device__ __forceinline__ void chain_finish(const Launch& L, const ChainTicket& c) {
    if ((threadIdx.x & 31) != 0) return;
    __threadfence();
    atomicMax(L.ch_done + c.item, c.strip + 1);
    if (L.ch_groups > 1) atomicAdd(L.ch_gdone + c.group, 1u);
    atomicAdd(L.ch_finished, 1);
}

// Polls of a wait for a column: every strip before this one may use up its own.
__device__ __forceinline__ uint32_t chain_polls(const Launch& L, int strip) {
    const unsigned long long p = static_cast<unsigned long long>(wait_polls(L)) * static_cast<unsigned long long>(strip + 1);
    return p > 0xfffffff0ull ? 0xfffffff0u : static_cast<uint32_t>(p);
}

}  // namespace sk
