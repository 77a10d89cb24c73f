// smem_cc.cuh -- connected components of one small graph by one thread block,
// the whole union-find in shared memory (Algorithm 1 without sampling on COO
// input): the batched kernel runs it per graph, the static COO call for graphs
// small enough for one block.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "uf_device.cuh"

namespace gc {

constexpr uint32_t SMEM_CAP = 1u << 20;   // loop cap of a thread's own union
// Cap of the turns that empty a warp's queue.  A queued pair's climb takes fewer
// than 2^18 turns: a turn lowers one of two ids below 2^16 or loses the one
// compare-and-swap that a root can lose.  So 160 pairs, at 32 a turn, are done in
// 5 x 2^18 turns; beyond the cap an invariant is broken.  (No measurable cost:
// 4,096 graphs 918-920 us without, 917-920 with it.)
constexpr uint32_t SMEM_TURNS = 1u << 21;

enum { BR_ASYNC_NAIVE = 0, BR_ASYNC_HALVE = 1, BR_REM_SPLIT = 2 };
constexpr int BATCH_ILP = 8;    // most rows of 32 edges a warp checks at a time
constexpr int BATCH_ROWS = 4;   // ... and queues before it drains
constexpr int BATCH_QUEUE = 32 + 32 * BATCH_ROWS;   // queued unions per warp (at most 31 left over)

template <class T>
__device__ __forceinline__ uint32_t sm_ld(const volatile T* P, uint32_t i) { return P[i]; }
__device__ __forceinline__ uint32_t sm_cas(volatile uint16_t* P, uint32_t i, uint32_t cmp, uint32_t val) {
    return atomicCAS((unsigned short*)(P + i), (unsigned short)cmp, (unsigned short)val);
}
__device__ __forceinline__ uint32_t sm_cas(volatile uint32_t* P, uint32_t i, uint32_t cmp, uint32_t val) {
    return atomicCAS((unsigned int*)(P + i), cmp, val);
}

template <int R, class T>
__device__ __forceinline__ uint32_t sm_find(volatile T* P, uint32_t u, uint32_t& left) {
    if constexpr (R == BR_ASYNC_HALVE) {
        while (left) {
            uint32_t v = sm_ld(P, u), w = sm_ld(P, v);
            if (v == w) return v;
            uint32_t old = sm_cas(P, u, v, w);
            u = old == v ? w : old;
            --left;
        }
        return u;
    } else {
        while (left) {
            uint32_t p = sm_ld(P, u);
            if (p == u) return u;
            u = p;
            --left;
        }
        return u;
    }
}

// One step of a Union-Rem-CAS climb with SplitAtomicOne (Algorithm 11) from
// the pair (u, v): true when the two sets are joined, else (u, v) is the pair
// to go on from.  Both cases of the step (link a root, split a path) run as one
// predicated sequence: a diverged warp would issue both branches, and the
// batched kernel is bound by instruction issue, not by shared-memory latency.
// The split is a plain store: w is an ancestor of ru, so a store that overtakes
// a newer one only leaves ru at an older ancestor, and a non-root never becomes
// a root (16-bit compare-and-swaps are emulated, several instructions each).
template <class T>
__device__ __forceinline__ bool sm_rem_step(volatile T* P, uint32_t& u, uint32_t& v) {
    const uint32_t a = sm_ld(P, u), b = sm_ld(P, v);
    const uint32_t hi = max(a, b), lo = min(a, b);
    const uint32_t ru = a < b ? v : u;
    bool done = hi == lo;
    const bool root = ru == hi;
    uint32_t w = hi;
    if (!done) w = sm_ld(P, hi);                                  // a root reads its own entry
    if (!done && !root && w != hi) P[ru] = (T)w;
    if (!done && root) done = sm_cas(P, ru, ru, lo) == ru;        // lost: ru has a parent now, go on from it
    v = a < b ? u : v;
    u = hi;
    return done;
}

// One whole Union-Async (naive or halving find, Algorithm 7) in shared memory.
template <int R, class T>
__device__ __forceinline__ void sm_union_async(volatile T* P, uint32_t u, uint32_t v, uint32_t* err) {
    uint32_t left = SMEM_CAP;
    uint32_t pu = sm_find<R, T>(P, u, left), pv = sm_find<R, T>(P, v, left);
    while (pu != pv && left) {
        if (pu < pv) { uint32_t t = pu; pu = pv; pv = t; }
        if (sm_ld(P, pu) == pu && sm_cas(P, pu, pu, pv) == pu) return;
        --left;
        pu = sm_find<R, T>(P, pu, left);
        pv = sm_find<R, T>(P, pv, left);
    }
    if (!left) atomicOr(err, GC_DERR_NONCONV);
}

// One whole union of a thread.
template <int R, class T>
__device__ __forceinline__ void sm_union(volatile T* P, uint32_t u, uint32_t v, uint32_t* err) {
    if constexpr (R == BR_REM_SPLIT) {
        for (uint32_t left = SMEM_CAP; left; --left)
            if (sm_rem_step<T>(P, u, v)) return;
        atomicOr(err, GC_DERR_NONCONV);
    } else {
        sm_union_async<R, T>(P, u, v, err);
    }
}

// Every vertex's root to global memory; all threads of the block, after their unions.
template <class T>
__device__ __forceinline__ void sm_labels(volatile T* P, uint32_t n, uint32_t* __restrict__ labels) {
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
        uint32_t r = i, left = SMEM_CAP;
        while (left--) {
            uint32_t p = sm_ld(P, r);
            if (p == r) break;
            r = p;
        }
        labels[i] = r;
    }
    __syncthreads();
}

// A large graph's edges mostly join nothing (a mean degree of 4 to 32 against
// one link per vertex), and a union of 32 edges in lock step takes as many
// steps as its longest climb.  So a warp first compares the parents of
// BATCH_ILP x 32 edges (equal parents: same set, done), packs the edges that
// differ into a queue in shared memory, and runs their climbs 32 at a time, ONE
// step per turn, putting the unfinished pairs back: the lanes stay full whatever
// the climbs' lengths, and every turn takes a climb further down, so the queue
// runs dry.  Ids are below 65,536, so a pair is one 32-bit word.
// The kernel is bound by instruction issue (about two steps an edge that links;
// the streaming alone takes 700 us of the batch), so what counts is the length
// of a step.  4,096 graphs (n log-uniform in [256, 65536], half ER, half RMAT,
// 434 M edges), default table: 1,322 -> 915 us (2.6 -> 3.8 TB/s on 8 bytes an
// edge).  The parts, in the order they were measured: the queue with whole
// climbs 1,256 us; a plain store for the split 1,213; eight, four, two steps a
// turn 1,212, 1,165, 1,103; the predicated step and 32-bit queue words 1,021;
// one step a turn 988.  Four rows checked at a time instead of eight 983, six
// 918; draining after each row instead of every four 997 (the drain is inlined
// once per place, and registers bound the co-resident classes).
//
// ILP rows of 32 edges a turn of a warp; 1: a union per thread, no queue.  What is
// left of a list below a turn of the block is spread over its warps row by row.
//
// Every thread of the block calls; smem holds smem_cc_bytes() bytes.
template <int R, class T, int ILP = BATCH_ILP>
__device__ __forceinline__ void smem_cc(uint32_t* smem, uint32_t n, const uint2* __restrict__ E, uint64_t m,
                                        uint32_t* __restrict__ labels, uint32_t* err) {
    constexpr int ROWS = ILP < BATCH_ROWS ? ILP : BATCH_ROWS;
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x / 32, lt = (1u << lane) - 1;
    uint32_t* uq = smem + warp * BATCH_QUEUE;    // the warps' union queues, then the parents
    volatile T* P = reinterpret_cast<volatile T*>(smem + (blockDim.x / 32) * BATCH_QUEUE);
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) P[i] = (T)i;
    __syncthreads();
    if constexpr (ILP == 1) {   // a union per thread, no queue
        for (uint64_t j = threadIdx.x; j < m; j += blockDim.x) {
            const uint2 e = __ldcs(E + j);
            if (e.x >= n || e.y >= n) atomicOr(err, GC_DERR_RANGE);
            else if (e.x != e.y) sm_union<R, T>(P, e.x, e.y, err);
        }
        __syncthreads();
        sm_labels(P, n, labels);
        return;
    }
    unsigned cnt = 0;        // the warp's queued unions
    auto drain = [&](unsigned take) {   // one turn of the last `take` (<= 32) queued pairs
        cnt -= take;
        bool more = false;
        uint32_t u = 0, v = 0;
        if (lane < take) {
            const uint32_t f = uq[cnt + lane];
            u = f & 0xFFFFu;
            v = f >> 16;
            if constexpr (R == BR_REM_SPLIT) more = !sm_rem_step<T>(P, u, v);
            else sm_union_async<R, T>(P, u, v, err);
        }
        const unsigned mk = __ballot_sync(0xFFFFFFFFu, more);
        if (more) uq[cnt + __popc(mk & lt)] = u | (v << 16);
        cnt += __popc(mk);
        __syncwarp();
    };
    auto drain_below = [&](unsigned low) {   // until fewer than `low` pairs are queued
        for (uint32_t left = SMEM_TURNS; cnt >= low; --left) {
            if (!left) {
                atomicOr(err, GC_DERR_NONCONV);
                cnt = 0;
                break;
            }
            drain(min(cnt, 32u));
        }
    };
    auto check = [&](uint2 (&e)[ILP]) {
        uint32_t top = 0;
#pragma unroll
        for (int k = 0; k < ILP; ++k) top = max(top, max(e[k].x, e[k].y));
        if (top >= n) {
            atomicOr(err, GC_DERR_RANGE);
#pragma unroll
            for (int k = 0; k < ILP; ++k)
                if (e[k].x >= n || e[k].y >= n) e[k] = make_uint2(0, 0);
        }
        uint32_t a[ILP], b[ILP];
#pragma unroll
        for (int k = 0; k < ILP; ++k) {
            a[k] = sm_ld(P, e[k].x);
            b[k] = sm_ld(P, e[k].y);
        }
#pragma unroll
        for (int h = 0; h < ILP; h += ROWS) {
#pragma unroll
            for (int k = h; k < h + ROWS; ++k) {
                const bool open = a[k] != b[k];
                const unsigned mk = __ballot_sync(0xFFFFFFFFu, open);
                if (open) uq[cnt + __popc(mk & lt)] = e[k].x | (e[k].y << 16);
                cnt += __popc(mk);
            }
            __syncwarp();
            drain_below(32);
        }
    };
    constexpr uint64_t PIECE = 1u << 30;   // edges per 32-bit index range
    const uint32_t B = blockDim.x;
    for (uint64_t m0 = 0; m0 < m; m0 += PIECE) {
        const uint32_t len = (uint32_t)(m - m0 < PIECE ? m - m0 : PIECE), full = len - len % (B * ILP);
        const uint2* Eg = E + m0 + lane;
        uint2 e[ILP];
        for (uint32_t j = warp * 32 * ILP; j < full; j += B * ILP) {
#pragma unroll
            for (int k = 0; k < ILP; ++k) e[k] = __ldcs(Eg + j + k * 32);
            check(e);
        }
        const uint32_t j = full + warp * 32;
        if (j < len) {   // less than a turn of the block
#pragma unroll
            for (int k = 0; k < ILP; ++k)
                e[k] = j + k * B + lane < len ? __ldcs(Eg + j + k * B) : make_uint2(0, 0);
            check(e);
        }
    }
    drain_below(1);
    __syncthreads();
    sm_labels(P, n, labels);
}

// Shared memory of one block for graphs of up to max_n vertices, and whether
// 32-bit parents fit beside the queues and the static words.
constexpr int SMEM_BLOCK_MAX = 227 * 1024 - 64;   // beside the kernels' static words
inline size_t smem_queue_bytes(int block) { return sizeof(uint32_t) * BATCH_QUEUE * (size_t)(block / 32); }
inline bool smem_wide(uint32_t max_n, int block) {
    return 4ull * max_n + smem_queue_bytes(block) <= (uint64_t)SMEM_BLOCK_MAX;
}
inline size_t smem_cc_bytes(uint32_t max_n, int block) {
    return smem_queue_bytes(block) + (smem_wide(max_n, block) ? sizeof(uint32_t) * (size_t)max_n
                                                              : sizeof(uint16_t) * (size_t)((max_n + 1) & ~1u));
}

}  // namespace gc
