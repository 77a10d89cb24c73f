// gconn_rounds.cu -- round-based finish algorithms: root-based
// Shiloach-Vishkin (Algorithm 12), the 16 Liu-Tarjan rule sets (appendix
// list), label propagation and Stergiou's algorithm, over a COO edge list,
// and the gather step that feeds them the arcs of the active CSR vertices.
//
// Each algorithm runs as ONE cooperative launch (every block resident) that
// loops over its rounds on the device: the phases of a round (an edge pass,
// vertex passes) are separated by grid barriers, a round that changes
// anything records its number in a control word, and every block reads that
// word after the round's last barrier to decide, identically, whether to run
// another round.  No host round trip per round, so these finishes can also be
// captured into a CUDA graph.  A grid barrier acquires at device scope, so what
// a phase does not write may be read through L1 in it; what other blocks write
// in the same phase is read through L2 (ld.global.cg), except where an older
// value serves as well (said at the place).
//
// What bounded the rounds: every edge's message was an atomic, and most aim at a
// few roots; RMAT n = 2^20, m = 2^24 on one GB300, SV / Liu-Tarjan PRF:
// 1,292 / 4,062-6,067 us at first; no atomic for a message that cannot win, finished
// edges left out of later rounds (for_live_edges) 605 / 1,034; what a block has
// sent already remembered in shared memory (SentTable), labels read through L1
// 375 / 696; compression walks through L1 350 / 629.  1024 x 1024 grid + 16
// paths of 65,536 (13 to 17 rounds): 864 / 1,064 -> 372 / 482 us, almost all of it the
// walks through L1.  Blocks per SM: 4, 5, 6, 8 within 2 % but 8 spills (LT 700).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "gc_internal.h"
#include "gc_static.h"
#include "static_kernels.cuh"

namespace gc {

constexpr unsigned long long NOMSG = 0xFFFFFFFFFFFFFFFFull;
constexpr uint32_t MAX_ROUNDS = 1u << 16;   // round cap: E_NONCONVERGED beyond it
constexpr int RB = 256;                     // block size of the round kernels

// Control words of one round kernel, zeroed before its launch.  chg only
// grows: after round r's last barrier every block reads it, and it is at
// least r + 1 exactly when round r changed something (a block that already
// went on to round r + 1 can only have raised it further).
struct RoundCtl {
    GridBar bar;
    uint32_t chg;      // 1 + the last round in which something changed
    uint32_t rounds;   // rounds run (written once, at the end)
    uint32_t pad[4];
};

__device__ __forceinline__ uint64_t gtid() { return (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; }
__device__ __forceinline__ uint64_t gstride() { return (uint64_t)gridDim.x * blockDim.x; }

// Records that round r changed something (one atomic per block); called by
// every thread of a block at the same point.
__device__ __forceinline__ void mark_changed(bool ch, uint32_t* chg, uint32_t r) {
    if (__syncthreads_or(ch) && threadIdx.x == 0) atomicMax(chg, r + 1);
}

// Whether round r changed anything, read after the round's last barrier:
// thread 0 reads the word once for the block.  The next round reaches
// another barrier (which synchronises the block) before it reads again.
__device__ __forceinline__ bool round_changed(const RoundCtl* ctl, uint32_t r) {
    __shared__ uint32_t s_chg;
    if (threadIdx.x == 0) s_chg = __ldcg(&ctl->chg);
    __syncthreads();
    return s_chg >= r + 1;
}

__device__ __forceinline__ uint64_t edge_count(uint64_t m_host, const unsigned long long* m_dev) {
    if (!m_dev) return m_host;
    unsigned long long m = __ldcg(m_dev);
    return m < m_host ? m : m_host;
}

// FullShortcut while nothing links: every vertex points at its root, and prev
// (optional) receives the same value.  The walk may read through L1: the grid
// barrier before this phase dropped what L1 held, roots rest, and an entry read
// before another thread shortened it is an older ancestor on the same path.
// One walk a thread: two or four in lock step wait for the longest (4 M-vertex
// grid + paths: 756, 802, 917 us of SV).
__device__ __forceinline__ void compress_copy(uint32_t n, uint32_t* P, uint32_t* prev, uint32_t* err) {
    for (uint64_t v = gtid(); v < n; v += gstride()) {
        uint32_t p = __ldcg(P + v), r = p;
        for (uint32_t i = 0;; ++i) {
            uint32_t q = __ldca(P + r);
            if (q == r) break;
            r = q;
            if (i == n) { atomicOr(err, GC_DERR_NONCONV); break; }
        }
        if (r != p) __stcg(P + v, r);
        if (prev) __stcg(prev + v, r);
    }
}

// The round cap: every block reaches it in the same round.
__device__ __forceinline__ bool over_cap(uint32_t r, uint32_t* err) {
    if (r < MAX_ROUNDS) return false;
    if (gtid() == 0) atomicOr(err, GC_DERR_NONCONV);
    return true;
}

__device__ __forceinline__ void finish_rounds(RoundCtl* ctl, uint32_t r) {
    if (gtid() == 0) ctl->rounds = r;
}

// ------------------------------------------------------------- edge passes
// The edges of one round, ROUND_ILP chunks of 32 a warp at a time, and the edges
// that are done left out.  body(i, e) gets arrays of ROUND_ILP edges (an edge
// that is not taken reads as (0, 0)) and sets keep[k] where edge k can still
// matter in a later round.
//
// live (one bit per edge, a word per chunk) remembers that: round 0 takes every
// edge and writes the words, later rounds read a word before the edge, so a
// chunk with no live edge costs a quarter sector instead of 8 of edges and 64 of
// labels.  A warp meets the same chunks in every round, so only it touches their
// words.  Null: every edge in every round.
constexpr int ROUND_ILP = 2;

template <class Body>
__device__ __forceinline__ void for_live_edges(const uint2* __restrict__ E, uint64_t m, uint32_t n, uint32_t* live,
                                               uint32_t r, uint32_t* err, Body&& body) {
    const unsigned lane = lane_id();
    const uint64_t chunks = (m + 31) / 32, nw = gstride() / 32;
    for (uint64_t c0 = gtid() / 32 * ROUND_ILP; c0 < chunks; c0 += nw * ROUND_ILP) {
        uint32_t w[ROUND_ILP], any = 0;
#pragma unroll
        for (int k = 0; k < ROUND_ILP; ++k) {
            w[k] = c0 + k >= chunks ? 0u : live && r ? live[c0 + k] : 0xFFFFFFFFu;
            any |= w[k];
        }
        if (!any) continue;
        uint2 e[ROUND_ILP];
        bool keep[ROUND_ILP];
#pragma unroll
        for (int k = 0; k < ROUND_ILP; ++k) {
            const uint64_t i = (c0 + k) * 32 + lane;
            e[k] = (w[k] >> lane & 1u) && i < m ? __ldcs(E + i) : make_uint2(0, 0);
        }
#pragma unroll
        for (int k = 0; k < ROUND_ILP; ++k)
            if (e[k].x >= n || e[k].y >= n) {
                atomicOr(err, GC_DERR_RANGE);
                e[k] = make_uint2(0, 0);
            }
        body(c0 * 32 + lane, e, keep);
        if (live)
#pragma unroll
            for (int k = 0; k < ROUND_ILP; ++k) {
                const uint32_t x = __ballot_sync(0xFFFFFFFFu, keep[k]);
                if (lane == 0 && c0 + k < chunks && (x != w[k] || r == 0)) live[c0 + k] = x;
            }
    }
}

// Every vertex that holds a message, which is taken from it; four loads in flight.
constexpr int MSG_ILP = 4;
template <class Body>
__device__ __forceinline__ void for_messages(uint32_t n, unsigned long long* msg, Body&& body) {
    for (uint64_t x0 = gtid(); x0 < n; x0 += gstride() * MSG_ILP) {
        unsigned long long mv[MSG_ILP];
#pragma unroll
        for (int j = 0; j < MSG_ILP; ++j) mv[j] = x0 + j * gstride() < n ? __ldcg(msg + x0 + j * gstride()) : NOMSG;
#pragma unroll
        for (int j = 0; j < MSG_ILP; ++j) {
            if (mv[j] == NOMSG) continue;
            msg[x0 + j * gstride()] = NOMSG;
            body(x0 + j * gstride(), mv[j]);
        }
    }
}

// What this block last sent to a receiver in the current round, one 64-bit word
// (receiver, value) per slot of a direct-mapped table in shared memory.  Once
// trees have grown, most edges of a round aim at a few roots; without this every
// one of them reads the same few L2 sectors, which serve about one request a
// clock.  A slot that another warp overwrites only costs a repeated message.
constexpr uint32_t SENT_SLOTS = 512;
// Fewer edges than this cannot crowd a receiver for long: they send at once, and
// the reads that spare an atomic would only lengthen the phase (n = 1,000,
// m = 3,000: SV 34.6 us without, 37.2 with them).
constexpr uint64_t SENT_MIN_EDGES = 1u << 16;
struct SentTable {
    unsigned long long w[SENT_SLOTS];
    __device__ __forceinline__ void clear() {   // the whole block, at the start of a round
        for (uint32_t i = threadIdx.x; i < SENT_SLOTS; i += blockDim.x) w[i] = NOMSG;
        __syncthreads();
    }
    // True when this block has sent `to` a value below val, or (ties) val itself.
    __device__ __forceinline__ bool covered(uint32_t to, uint32_t val, bool ties) const {
        const unsigned long long x = *(volatile const unsigned long long*)&w[to & (SENT_SLOTS - 1)];
        const uint32_t v = (uint32_t)x;
        return (uint32_t)(x >> 32) == to && (v < val || (ties && v == val));
    }
    __device__ __forceinline__ void note(uint32_t to, uint32_t val) {
        *(volatile unsigned long long*)&w[to & (SENT_SLOTS - 1)] = ((unsigned long long)to << 32) | val;
    }
};

// --------------------------------------------------------------------- SV
// Shiloach-Vishkin (Algorithm 12), root-based.  Per round: the hook pass --
// for each edge the larger of its two current labels is writeMin'ed with the
// smaller when it was a root at round start (prev); forest form: each
// round-start root keeps the smallest (label, edge id) message, applied in a
// vertex pass -- then full compression, which also copies the labels into
// prev.  Stop after a round that hooked nothing.
template <bool SF>
__global__ void __launch_bounds__(RB, 6) k_sv(const uint2* __restrict__ E, const uint32_t* eids, uint64_t m_host,
                                           const unsigned long long* m_dev, uint32_t n, uint32_t* P, uint32_t* prev,
                                           unsigned long long* msg, uint32_t* sf, uint32_t* live, uint32_t* err,
                                           RoundCtl* ctl) {
    const uint64_t m = edge_count(m_host, m_dev);
    compress_copy(n, P, prev, err);
    if (SF)
        for (uint64_t x = gtid(); x < n; x += gstride()) msg[x] = NOMSG;
    __shared__ SentTable sent;
    const bool crowded = m >= SENT_MIN_EDGES;
    if (!grid_sync(&ctl->bar, err)) return;
    for (uint32_t r = 0;; ++r) {
        if (over_cap(r, err)) return;
        bool ch = false;
        if (crowded) sent.clear();
        for_live_edges(E, m, n, live, r, err, [&](uint64_t i0, uint2 (&e)[ROUND_ILP], bool (&keep)[ROUND_ILP]) {
            uint32_t lo[ROUND_ILP], hi[ROUND_ILP];
#pragma unroll
            for (int k = 0; k < ROUND_ILP; ++k) {
                // prev is not written in this phase, and a label of P that L1
                // holds from earlier in it is a label of the same tree
                const uint32_t* L = SF ? prev : P;
                const uint32_t pu = __ldca(L + e[k].x), pv = __ldca(L + e[k].y);
                lo[k] = min(pu, pv);
                hi[k] = max(pu, pv);
            }
#pragma unroll
            for (int k = 0; k < ROUND_ILP; ++k) {
                keep[k] = lo[k] != hi[k];   // one tree stays one tree
                if (!keep[k] || (crowded && sent.covered(hi[k], lo[k], !SF))) continue;
                if (crowded) sent.note(hi[k], lo[k]);
                if (SF) {
                    const uint64_t i = i0 + 32 * k;
                    const unsigned long long mv = ((unsigned long long)lo[k] << 32) | (eids ? eids[i] : (uint32_t)i);
                    if (!crowded || __ldcg(msg + hi[k]) > mv) atomicMin(msg + hi[k], mv);
                } else if ((!crowded || __ldcg(P + hi[k]) > lo[k]) && __ldcg(prev + hi[k]) == hi[k]) {
                    // (whoever lowered P[hi] this round to lo or below marked the change)
                    atomicMin(P + hi[k], lo[k]);
                    ch = true;
                }
            }
        });
        if (!SF) mark_changed(ch, &ctl->chg, r);
        if (!grid_sync(&ctl->bar, err)) return;
        if (SF) {   // apply the winning messages to round-start roots
            for_messages(n, msg, [&](uint64_t x, unsigned long long mv) {
                uint32_t val = (uint32_t)(mv >> 32);
                if (__ldcg(P + x) == (uint32_t)x && val < (uint32_t)x) {
                    __stcg(P + x, val);
                    sf[x] = (uint32_t)mv;
                    ch = true;
                }
            });
            mark_changed(ch, &ctl->chg, r);
            if (!grid_sync(&ctl->bar, err)) return;
        }
        compress_copy(n, P, prev, err);
        if (!grid_sync(&ctl->bar, err)) return;
        if (!round_changed(ctl, r)) {   // no change in round r (chg only grows)
            finish_rounds(ctl, r + 1);
            return;
        }
    }
}

// --------------------------------------------------------------------- LT
// One Liu-Tarjan rule set per launch (runtime flags).  Per round: Connect
// messages from the round-start parents go to msg by atomicMin (packed with
// the edge id for forests):
//   C: u receives v, v receives u
//   P: P[u] receives P[v], P[v] receives P[u]
//   E: u, v, P[u], P[v] all receive min(P[u], P[v])
// then Update (all vertices) or RootUpdate (round-start roots only), then one
// Shortcut jump per vertex or FullShortcut, then Alter (edge <- (P[u], P[v]),
// dropped when the ends meet).  Stop after a round that changes neither a
// parent nor an edge; then full compression.
__global__ void __launch_bounds__(RB, 6) k_lt(const uint2* __restrict__ E_in, uint2* Ew, const uint32_t* eids,
                                           uint64_t m_host, const unsigned long long* m_dev, uint32_t n, uint32_t* P,
                                           unsigned long long* msg, uint32_t* sf, uint32_t* live, int conn,
                                           int root_only, int full, uint32_t* err, RoundCtl* ctl) {
    const uint64_t m = edge_count(m_host, m_dev);
    const bool alter = Ew != nullptr;
    __shared__ SentTable sent;
    const bool crowded = m >= SENT_MIN_EDGES;
    for (uint64_t x = gtid(); x < n; x += gstride()) msg[x] = NOMSG;
    if (!grid_sync(&ctl->bar, err)) return;
    for (uint32_t r = 0;; ++r) {
        if (over_cap(r, err)) return;
        bool ch = false;
        // Connect.  Every parent is at or below its vertex, so a message that is
        // not below its receiver is never applied, and one that is not below what
        // the receiver already holds changes nothing: neither needs the atomic.
        if (crowded) sent.clear();
        auto send = [&](uint32_t to, uint32_t val, unsigned long long id) {
            if (val >= to || (crowded && sent.covered(to, val, !sf))) return;   // (a forest keeps the smallest edge id)
            if (crowded) sent.note(to, val);
            const unsigned long long mv = ((unsigned long long)val << 32) | id;
            if (!crowded || __ldcg(msg + to) > mv) atomicMin(msg + to, mv);
        };
        if (conn == GCONN_LT_PARENT && !alter) {
            for_live_edges(E_in, m, n, live, r, err, [&](uint64_t i0, uint2 (&e)[ROUND_ILP], bool (&keep)[ROUND_ILP]) {
                uint32_t lo[ROUND_ILP], hi[ROUND_ILP];
#pragma unroll
                for (int k = 0; k < ROUND_ILP; ++k) {
                    const uint32_t pu = __ldca(P + e[k].x), pv = __ldca(P + e[k].y);   // P rests here
                    lo[k] = min(pu, pv);
                    hi[k] = max(pu, pv);
                }
#pragma unroll
                for (int k = 0; k < ROUND_ILP; ++k) {
                    keep[k] = lo[k] != hi[k];
                    const uint64_t i = i0 + 32 * k;
                    if (keep[k]) send(hi[k], lo[k], eids ? eids[i] : (uint32_t)i);
                }
            });
        } else {
            for (uint64_t i = gtid(); i < m; i += gstride()) {
                uint2 e = alter ? __ldcg(Ew + i) : E_in[i];
                if (e.x == GC_DINF) continue;                   // dropped by Alter
                if (e.x >= n || e.y >= n) { atomicOr(err, GC_DERR_RANGE); continue; }
                if (e.x == e.y) continue;
                const unsigned long long id = eids ? eids[i] : (uint32_t)i;
                if (conn == GCONN_LT_CONNECT) {
                    send(e.x, e.y, id);
                    send(e.y, e.x, id);
                } else {
                    uint32_t pu = __ldcg(P + e.x), pv = __ldcg(P + e.y);
                    if (pu == pv) continue;
                    if (conn == GCONN_LT_PARENT) {
                        send(pu, pv, id);
                        send(pv, pu, id);
                    } else {
                        const uint32_t lo = min(pu, pv);
                        send(e.x, lo, id);
                        send(e.y, lo, id);
                        send(pu, lo, id);
                        send(pv, lo, id);
                    }
                }
            }
        }
        if (!grid_sync(&ctl->bar, err)) return;
        for_messages(n, msg, [&](uint64_t x, unsigned long long mv) {   // Update / RootUpdate
            uint32_t p = __ldcg(P + x), val = (uint32_t)(mv >> 32);
            if (root_only && p != (uint32_t)x) return;
            if (val < p) {
                __stcg(P + x, val);
                if (sf) sf[x] = (uint32_t)mv;
                ch = true;
            }
        });
        mark_changed(ch, &ctl->chg, r);
        if (!grid_sync(&ctl->bar, err)) return;
        ch = false;
        if (full) {
            compress_copy(n, P, nullptr, err);
        } else {                                                // one jump, in place
            for (uint64_t x = gtid(); x < n; x += gstride()) {
                uint32_t p = __ldcg(P + x), g2 = __ldcg(P + p);
                if (g2 != p) {
                    __stcg(P + x, g2);
                    ch = true;
                }
            }
            mark_changed(ch, &ctl->chg, r);
        }
        if (!grid_sync(&ctl->bar, err)) return;
        if (alter) {
            ch = false;
            for (uint64_t i = gtid(); i < m; i += gstride()) {
                uint2 e = __ldcg(Ew + i);
                if (e.x == GC_DINF) continue;
                uint2 f = make_uint2(__ldcg(P + e.x), __ldcg(P + e.y));
                if (f.x == f.y) f = make_uint2(GC_DINF, GC_DINF);
                if (f.x != e.x || f.y != e.y) {
                    __stcg(Ew + i, f);
                    ch = true;
                }
            }
            mark_changed(ch, &ctl->chg, r);
            if (!grid_sync(&ctl->bar, err)) return;
        }
        if (!round_changed(ctl, r)) {   // no change in round r (chg only grows)
            finish_rounds(ctl, r + 1);
            break;
        }
    }
    compress_copy(n, P, nullptr, err);
}

// --------------------------------------------------------------------- LP
// Label Propagation: per round, for each edge the larger endpoint label takes
// the smaller (atomicMin on both ends); stop after a round that changes
// nothing; then full compression.
__global__ void __launch_bounds__(RB) k_lp(const uint2* __restrict__ E, uint64_t m_host,
                                           const unsigned long long* m_dev, uint32_t n, uint32_t* P, uint32_t* err,
                                           RoundCtl* ctl) {
    const uint64_t m = edge_count(m_host, m_dev);
    for (uint32_t r = 0; m; ++r) {
        if (over_cap(r, err)) return;
        bool ch = false;
        for (uint64_t i = gtid(); i < m; i += gstride()) {
            uint2 e = E[i];
            if (e.x >= n || e.y >= n) { atomicOr(err, GC_DERR_RANGE); continue; }
            uint32_t a = __ldcg(P + e.x), b = __ldcg(P + e.y);
            if (a == b) continue;
            uint32_t lo = min(a, b);
            if (a > lo) atomicMin(P + e.x, lo);
            if (b > lo) atomicMin(P + e.y, lo);
            ch = true;
        }
        mark_changed(ch, &ctl->chg, r);
        if (!grid_sync(&ctl->bar, err)) return;
        if (!round_changed(ctl, r)) {   // no change in round r (chg only grows)
            finish_rounds(ctl, r + 1);
            break;
        }
    }
    compress_copy(n, P, nullptr, err);
}

// ---------------------------------------------------------------- Stergiou
// Per round: for each edge the entry of the larger of prev[u], prev[v]
// receives the smaller (atomicMin into the current labels), then one
// shortcut jump per vertex; the round changed something if a jump moved or a
// label differs from prev.  The shortcut pass also writes the next round's
// prev (each entry is written there by its own thread only).
__global__ void __launch_bounds__(RB) k_stergiou(const uint2* __restrict__ E, uint64_t m_host,
                                                 const unsigned long long* m_dev, uint32_t n, uint32_t* P,
                                                 uint32_t* prev, uint32_t* err, RoundCtl* ctl) {
    const uint64_t m = edge_count(m_host, m_dev);
    for (uint64_t x = gtid(); x < n; x += gstride()) prev[x] = __ldcg(P + x);
    if (!grid_sync(&ctl->bar, err)) return;
    for (uint32_t r = 0; m; ++r) {
        if (over_cap(r, err)) return;
        for (uint64_t i = gtid(); i < m; i += gstride()) {
            uint2 e = E[i];
            if (e.x >= n || e.y >= n) { atomicOr(err, GC_DERR_RANGE); continue; }
            uint32_t a = __ldcg(prev + e.x), b = __ldcg(prev + e.y);
            if (a == b) continue;
            const uint32_t lo = min(a, b), hi = max(a, b);
            if (m < SENT_MIN_EDGES || __ldcg(P + hi) > lo) atomicMin(P + hi, lo);
        }
        if (!grid_sync(&ctl->bar, err)) return;
        bool ch = false;
        for (uint64_t x = gtid(); x < n; x += gstride()) {
            uint32_t p = __ldcg(P + x), g2 = __ldcg(P + p);
            if (g2 != p) {
                __stcg(P + x, g2);
                ch = true;
            }
            if (__ldcg(prev + x) != g2) ch = true;
            __stcg(prev + x, g2);
        }
        mark_changed(ch, &ctl->chg, r);
        if (!grid_sync(&ctl->bar, err)) return;
        if (!round_changed(ctl, r)) {   // no change in round r (chg only grows)
            finish_rounds(ctl, r + 1);
            break;
        }
    }
    compress_copy(n, P, nullptr, err);
}

// ------------------------------------------------------------- CSR gather
struct Gather {
    uint2* E;
    uint32_t* ids;
    unsigned long long* cnt;
    unsigned long long cap;
};

__device__ __forceinline__ void gather_arc(const Gather& g, uint32_t u, uint32_t v, uint32_t a) {
    unsigned long long k = atomicAdd(g.cnt, 1ull);
    if (k < g.cap) {
        g.E[k] = make_uint2(u, v);
        g.ids[k] = a;
    }
}

template <class OffT>
__global__ void k_gather_small(const OffT* off, const uint32_t* cols, uint32_t n, const uint32_t* active,
                               const uint32_t* small, const uint32_t* nsmall, Gather g, uint32_t* err) {
    uint32_t cnt = *nsmall;
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += stride) {
        uint32_t u = small[i];
        for (uint64_t a = off[u]; a < off[u + 1]; ++a) {
            uint32_t v = cols[a];
            if (v >= n) { atomicOr(err, GC_DERR_RANGE); continue; }
            if (arc_needed(active, u, v)) gather_arc(g, u, v, (uint32_t)a);
        }
    }
}

template <class OffT>
__global__ void k_gather_tasks(const OffT* off, const uint32_t* cols, uint32_t n, const uint32_t* active,
                               const unsigned long long* tasks, const uint32_t* ntasks, uint32_t task_cap, Gather g,
                               uint32_t* err) {
    uint32_t cnt = min(*ntasks, task_cap);
    uint64_t nw = (uint64_t)gridDim.x * (blockDim.x / 32);
    unsigned lane = threadIdx.x & 31u;
    for (uint64_t t = (uint64_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32; t < cnt; t += nw) {
        unsigned long long task = tasks[t];
        uint32_t u = (uint32_t)(task >> 32);
        uint64_t lo = off[u] + (task & 0xFFFFFFFFull) * TASK_ARCS, hi = off[u + 1];
        if (lo + TASK_ARCS < hi) hi = lo + TASK_ARCS;
        for (uint64_t a = lo + lane; a < hi; a += 32) {
            uint32_t v = cols[a];
            if (v >= n) { atomicOr(err, GC_DERR_RANGE); continue; }
            if (arc_needed(active, u, v)) gather_arc(g, u, v, (uint32_t)a);
        }
    }
}

template <class OffT>
__global__ void k_gather_over(const OffT* off, const uint32_t* cols, uint32_t n, const uint32_t* active,
                              const uint32_t* over, const uint32_t* nover, Gather g, uint32_t* err) {
    uint64_t cnt = *nover;
    for (uint64_t i = blockIdx.x; i < cnt; i += gridDim.x) {
        uint32_t u = over[i];
        for (uint64_t a = off[u] + threadIdx.x; a < off[u + 1]; a += blockDim.x) {
            uint32_t v = cols[a];
            if (v >= n) { atomicOr(err, GC_DERR_RANGE); continue; }
            if (arc_needed(active, u, v)) gather_arc(g, u, v, (uint32_t)a);
        }
    }
}

// ------------------------------------------------------------------ drivers
// Scratch for one round kernel: its control words (zeroed on the stream).
struct RoundLaunch {
    DevBuf ctlb;
    RoundCtl* ctl = nullptr;
    gconn_status init(cudaStream_t st) {
        GC_TRY(ctlb.alloc(sizeof(RoundCtl), st));
        ctl = ctlb.as<RoundCtl>();
        GC_CUDA(cudaMemsetAsync(ctl, 0, sizeof(RoundCtl), st));
        return GCONN_OK;
    }
    // Rounds run, for the edge-pass count (waits for the stream).
    gconn_status rounds(cudaStream_t st, uint32_t* out) {
        uint32_t r = 0;
        GC_CUDA(cudaMemcpyAsync(&r, &ctl->rounds, sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
        GC_CUDA(cudaStreamSynchronize(st));
        *out = r;
        return GCONN_OK;
    }
};

// One bit per edge for for_live_edges.  Only a saving: a list that the GPU reads
// in one go does without, and without the memory for it (m / 8 bytes) every
// round reads every edge.  A captured pass does without too: there the allocation
// is a node of the plan, and where it does not fit the whole plan fails.
static uint32_t* live_bits(DevBuf& buf, uint64_t m, cudaStream_t st) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (m < SENT_MIN_EDGES || cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone)
        return nullptr;
    if (buf.alloc(sizeof(uint32_t) * ((m + 31) / 32), st) != GCONN_OK) return nullptr;
    return buf.as<uint32_t>();
}

template <class K>
unsigned round_grid(K kernel, uint64_t m, uint32_t n) {
    return grid_for(kernel, RB, std::max<uint64_t>(m, n));
}

static gconn_status run_sv(const UFState& s, const uint2* E, const uint32_t* eids, uint64_t m,
                           const unsigned long long* m_dev, cudaStream_t st, uint32_t* rounds) {
    uint32_t n = s.n;
    DevBuf prevb, msgb;
    GC_TRY(prevb.alloc(sizeof(uint32_t) * (size_t)n, st));
    unsigned long long* msg = nullptr;
    bool sf = s.sf != nullptr;
    if (sf) {
        GC_TRY(msgb.alloc(sizeof(unsigned long long) * (size_t)n, st));
        msg = msgb.as<unsigned long long>();
    }
    RoundLaunch rl;
    GC_TRY(rl.init(st));
    DevBuf liveb;
    // (a caller that counts edge inspections is told of every round's whole pass)
    uint32_t* live = rounds ? nullptr : live_bits(liveb, m, st);
    auto k = sf ? k_sv<true> : k_sv<false>;
    GC_TRY(launch_coop("sv", k, round_grid(k, m, n), RB, 0, st, E, eids, m, m_dev, n, s.P, prevb.as<uint32_t>(), msg,
                       s.sf, live, s.err, rl.ctl));
    return rounds ? rl.rounds(st, rounds) : GCONN_OK;
}

static gconn_status run_lt(const Variant& v, const UFState& s, const uint2* E_in, const uint32_t* eids, uint64_t m,
                           const unsigned long long* m_dev, cudaStream_t st, uint32_t* rounds) {
    uint32_t n = s.n;
    int conn = v.lt_rules & 3;
    bool root_only = (v.lt_rules & GCONN_LT_ROOTUPDATE) != 0;
    bool full = (v.lt_rules & GCONN_LT_FULLSHORTCUT) != 0;
    bool alter = (v.lt_rules & GCONN_LT_ALTER) != 0;
    DevBuf msgb, eb;
    GC_TRY(msgb.alloc(sizeof(unsigned long long) * (size_t)n, st));
    uint2* Ew = nullptr;
    if (alter && m) {   // Alter rewrites the edges: work on a copy
        GC_TRY(eb.alloc(sizeof(uint2) * m, st));
        Ew = eb.as<uint2>();
        GC_CUDA(cudaMemcpyAsync(Ew, E_in, sizeof(uint2) * m, cudaMemcpyDeviceToDevice, st));
    }
    RoundLaunch rl;
    GC_TRY(rl.init(st));
    // With ParentConnect and FullShortcut two vertices that share a parent share
    // it for good (parents are roots, and members follow their root), so their
    // edge is done.  Other rules can part them again.
    DevBuf liveb;
    uint32_t* live = conn == GCONN_LT_PARENT && full && !alter && !rounds ? live_bits(liveb, m, st) : nullptr;
    GC_TRY(launch_coop("lt", k_lt, round_grid(k_lt, m, n), RB, 0, st, E_in, Ew, eids, m, m_dev, n, s.P,
                       msgb.as<unsigned long long>(), s.sf, live, conn, (int)root_only, (int)full, s.err, rl.ctl));
    if (!rounds) return GCONN_OK;
    GC_TRY(rl.rounds(st, rounds));
    *rounds *= (m ? 1u : 0u) + (alter && m ? 1u : 0u);   // connect (+ alter) read every edge
    return GCONN_OK;
}

static gconn_status run_lp(const UFState& s, const uint2* E, uint64_t m, const unsigned long long* m_dev,
                           cudaStream_t st, uint32_t* rounds) {
    RoundLaunch rl;
    GC_TRY(rl.init(st));
    GC_TRY(launch_coop("lp", k_lp, round_grid(k_lp, m, s.n), RB, 0, st, E, m, m_dev, s.n, s.P, s.err, rl.ctl));
    return rounds ? rl.rounds(st, rounds) : GCONN_OK;
}

static gconn_status run_stergiou(const UFState& s, const uint2* E, uint64_t m, const unsigned long long* m_dev,
                                 cudaStream_t st, uint32_t* rounds) {
    DevBuf prevb;
    GC_TRY(prevb.alloc(sizeof(uint32_t) * (size_t)s.n, st));
    RoundLaunch rl;
    GC_TRY(rl.init(st));
    GC_TRY(launch_coop("stergiou", k_stergiou, round_grid(k_stergiou, m, s.n), RB, 0, st, E, m, m_dev, s.n, s.P,
                       prevb.as<uint32_t>(), s.err, rl.ctl));
    return rounds ? rl.rounds(st, rounds) : GCONN_OK;
}

gconn_status rounds_coo(const Variant& v, const UFState& s, const uint32_t* edges, const uint32_t* eids, uint64_t m,
                        cudaStream_t st, uint32_t* edge_passes, const unsigned long long* m_dev) {
    uint32_t passes = 0;
    uint32_t* pp = edge_passes ? &passes : nullptr;
    gconn_status r = GCONN_OK;
    const uint2* E = (const uint2*)edges;
    if (s.n == 0) r = GCONN_OK;
    else if (v.link == GCONN_LINK_SV) r = run_sv(s, E, eids, m, m_dev, st, pp);
    else if (v.link == GCONN_LINK_LP) r = run_lp(s, E, m, m_dev, st, pp);
    else if (v.link == GCONN_LINK_STERGIOU) r = run_stergiou(s, E, m, m_dev, st, pp);
    else r = run_lt(v, s, E, eids, m, m_dev, st, pp);
    if (edge_passes) *edge_passes = passes;
    return r;
}

template <class OffT>
gconn_status rounds_csr(const Variant& v, const UFState& s, const OffT* off, const uint32_t* cols,
                        const uint32_t* active, const uint32_t* small, const uint32_t* nsmall,
                        const unsigned long long* tasks, const uint32_t* ntasks, uint32_t task_cap,
                        const uint32_t* over, const uint32_t* nover, cudaStream_t st) {
    uint32_t n = s.n;
    // the gathered arcs are at most all arcs: the host needs offsets[n] to
    // size the list (known in advance while a plan is being captured)
    uint64_t narcs = csr_arcs_hint();
    if (narcs == UINT64_MAX) {
        OffT last = 0;
        GC_CUDA(cudaMemcpyAsync(&last, off + n, sizeof(OffT), cudaMemcpyDeviceToHost, st));
        GC_CUDA(cudaStreamSynchronize(st));
        narcs = last;
    }
    DevBuf eb, ib, cb;
    uint64_t cap = narcs ? narcs : 1;
    GC_TRY(eb.alloc(sizeof(uint2) * cap, st));
    GC_TRY(ib.alloc(sizeof(uint32_t) * cap, st));
    GC_TRY(cb.alloc(sizeof(unsigned long long), st));
    Gather g{eb.as<uint2>(), ib.as<uint32_t>(), cb.as<unsigned long long>(), cap};
    GC_CUDA(cudaMemsetAsync(g.cnt, 0, sizeof(unsigned long long), st));
    GC_TRY(launch("gather_small", k_gather_small<OffT>, grid_for(k_gather_small<OffT>, 256, n), 256, 0, st, off,
                  cols, n, active, small, nsmall, g, s.err));
    GC_TRY(launch("gather_tasks", k_gather_tasks<OffT>, grid_for(k_gather_tasks<OffT>, 256, (uint64_t)n * 32), 256,
                  0, st, off, cols, n, active, tasks, ntasks, task_cap, g, s.err));
    GC_TRY(launch("gather_over", k_gather_over<OffT>, grid_for(k_gather_over<OffT>, 256, (uint64_t)n * 256), 256, 0,
                  st, off, cols, n, active, over, nover, g, s.err));
    // the rounds read the gathered count on the device
    return rounds_coo(v, s, (const uint32_t*)g.E, g.ids, cap, st, nullptr, g.cnt);
}

template gconn_status rounds_csr<uint32_t>(const Variant&, const UFState&, const uint32_t*, const uint32_t*,
                                          const uint32_t*, const uint32_t*, const uint32_t*,
                                          const unsigned long long*, const uint32_t*, uint32_t, const uint32_t*,
                                          const uint32_t*, cudaStream_t);
template gconn_status rounds_csr<uint64_t>(const Variant&, const UFState&, const uint64_t*, const uint32_t*,
                                          const uint32_t*, const uint32_t*, const uint32_t*,
                                          const unsigned long long*, const uint32_t*, uint32_t, const uint32_t*,
                                          const uint32_t*, cudaStream_t);

}  // namespace gc
