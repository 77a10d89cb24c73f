// gconn_coo.cu -- the union-find finish over a COO edge list: static passes
// (Algorithm 1 on COO input, Section 2) and insert batches (Section 3.5).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "csr_impl.cuh"
#include "gc_internal.h"
#include "gc_static.h"
#include "smem_cc.cuh"
#include "static_kernels.cuh"

namespace gc {

template <int R>
static __global__ void __launch_bounds__(1024, 1) k_small_cc(uint32_t n, const uint2* __restrict__ E, uint32_t m,
                                                             uint32_t* __restrict__ labels, uint32_t* err) {
    pdl_entry();
    extern __shared__ uint32_t smem_raw[];
    smem_cc<R, uint32_t, 2>(smem_raw, n, E, m, labels, err);
}

// The whole static pass of a small COO graph in one block, with the variant's
// own rule (the three that smem_cc has); *done says whether the call took it.
// Three dependent kernels cost their launch gaps and L2 round trips whatever
// the size; one block walks 32 edges a turn per warp in shared memory.  The
// limits, by rule (microseconds of the kernels in a captured plan, three kernels
// -> one block):
// - Rem-CAS climbs one step a turn with full lanes: n = 1,000, m = 4,000 16 -> 8,
//   m = 64,000 27 -> 18; n = 16,384, m = 32,768 36 -> 30 (ER), 22 -> 18 (RMAT),
//   m = 65,536 43 -> 36, 33 -> 25; m = 128,000 no gain.
// - Union-Async runs a whole union per lane, so a turn takes as long as its longest
//   walk.  Halving keeps the walks short: n = 4,096, m = 4,096 21 -> 13, m = 65,536
//   37 -> 28; but n = 16,384, m = 32,768 29 -> 41.  Naive walks grow with the
//   list: n = 1,000, m = 1,000 14 -> 10, m = 4,000 18 -> 20; n = 4,096, m = 16,384
//   23 -> 53.
// Host lists are read in place over the host link, by this one SM: wall time a
// call, page-locked, n = 16,384: Rem-CAS m = 32,768 57 -> 57, m = 65,536 67 -> 71;
// halving n = 4,096, m = 16,384 43 -> 42, m = 32,768 47 -> 48.
// A caller's own iteration cap counts the steps of the global-memory rules, and a
// caller's own block size is meant for them: those calls keep them.
struct SmallLimit {
    uint32_t n, m, m_host;
};
static SmallLimit small_limit(int rule) {
    return rule == BR_REM_SPLIT ? SmallLimit{16384, 65536, 32768}
         : rule == BR_ASYNC_HALVE ? SmallLimit{4096, 65536, 16384} : SmallLimit{16384, 1024, 1024};
}

gconn_status small_cc(const Variant& v, const UFState& s, const uint32_t* edges, uint64_t m, bool host,
                      cudaStream_t st, bool* done) {
    *done = false;
    if (v.cap != DEFAULT_CAP || v.block > 0) return GCONN_OK;
    int L, F, S;
    uf_triple(v, &L, &F, &S);
    const int rule = L == LK_REMCAS && F == FD_NAIVE && S == SP_SPLIT_ONE ? BR_REM_SPLIT
                   : L == LK_ASYNC && F == FD_NAIVE ? BR_ASYNC_NAIVE
                   : L == LK_ASYNC && F == FD_HALVE ? BR_ASYNC_HALVE : -1;
    if (rule < 0) return GCONN_OK;
    const SmallLimit lim = small_limit(rule);
    if (s.n > lim.n || m > (host ? lim.m_host : lim.m)) return GCONN_OK;
    auto k = rule == BR_REM_SPLIT ? k_small_cc<BR_REM_SPLIT>
           : rule == BR_ASYNC_NAIVE ? k_small_cc<BR_ASYNC_NAIVE> : k_small_cc<BR_ASYNC_HALVE>;
    const int B = 1024;
    const size_t smem = smem_cc_bytes(s.n, B);
    // always the rule's largest size: calls from several threads share the attribute
    GC_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_cc_bytes(lim.n, B)));
    *done = true;
    return launch_pdl("small_cc", k, 1, B, smem, st, s.n, (const uint2*)edges, (uint32_t)m, s.P, s.err);
}

gconn_status union_coo(const Variant& v, const UFState& s, const uint32_t* edges, uint64_t m,
                       uint32_t eid_base, cudaStream_t st) {
    if (m == 0) return GCONN_OK;
    int L, F, S;
    uf_triple(v, &L, &F, &S);
    int B = block_of(v);
    return dispatch_uf(L, F, S, s.sf != nullptr, [&]<int l, int f, int sp, bool sf>() {
        auto k = k_union_coo<l, f, sp, sf>;
        // at most about one thread per vertex: beyond that, concurrent unions
        // on a small vertex set mostly contend for the same few roots (ER
        // n = 65,536, m = 2^20, Rem-CAS + splice: 0.140 ms with the full
        // grid, 0.097 ms with a quarter of it, 0.116 ms with an eighth)
        uint64_t gr = grid_for(k, B, m);
        const uint64_t cap = std::max<uint64_t>((uint64_t)num_sms(), ((uint64_t)s.n + B - 1) / B);
        return launch_pdl("union_coo", k, (unsigned)std::min(gr, cap), B, 0, st, (const uint2*)edges, m, s, eid_base);
    });
}

// The COO finish of a static pass (every vertex a singleton at the start).
// Three forms, by size:
// - fewer edges than fill the GPU once (m < 49,152): one union per thread;
//   comparing first only adds a round trip (ER n = 16,000, m = 32,000: 34 against
//   53 us).
// - 2^15 <= n <= 2^19 and m >= 2n: as many threads as vertices or more would
//   start on singletons at once and contend for the same few roots.  So about
//   3n/4 edges, spread over the list, are united first (where a random graph's
//   giant component appears), the trees are flattened, and the other edges then
//   mostly find equal parents.  ER n = 65,536, m = 2^20: 98 -> 49 us (85 without
//   the first pass; a sample of n/2 or n edges 80, 50); n = 200,000, m = 16n:
//   168 -> 80 (98); RMAT n = 400,000, m = 8n: 144 -> 82 (84).  Above 2^19 the
//   first wave no longer covers the vertices (RMAT n = 10^6: 156 us without,
//   173 with); at 16,000 vertices the two launches cost what they save (45, 48).
// - otherwise one pass over all edges.
gconn_status union_coo_static(const Variant& v, const UFState& s, const uint32_t* edges, uint64_t m, cudaStream_t st) {
    if (v.link == GCONN_LINK_JTB || m < 49152) return union_coo(v, s, edges, m, 0, st);
    int L, F, S;
    uf_triple(v, &L, &F, &S);
    const int B = block_of(v);
    const uint64_t n = s.n;
    return dispatch_uf(L, F, S, s.sf != nullptr, [&]<int l, int f, int sp, bool sf>() -> gconn_status {
        if constexpr (l == LK_JTB) return GCONN_E_UNSUPPORTED;   // handled above
        else {
            auto pass = [&](const char* name, bool dense, CooPart part, uint64_t count) {
                auto k = dense ? k_union_filter<l, f, sp, sf, 8> : k_union_filter<l, f, sp, sf, 2>;
                return launch_pdl(name, k, grid_for(k, B, count / (dense ? 8 : 2) + 1), B, 0, st, (const uint2*)edges,
                                  m, s, part);
            };
            const bool dense = m >= 4 * n;   // most edges join nothing
            // rules that compress nothing on the way (naive finds of
            // Union-Async and Union-Hooks, Afforest)
            constexpr bool bare = rule_is_bare<l, f>();
            if (bare && n < (1u << 15)) return union_coo(v, s, edges, m, 0, st);
            if (n >= (1u << 15) && (bare || n <= (1u << 19)) && m >= 2 * n) {
                const uint32_t every = (uint32_t)std::min<uint64_t>(4 * m / (3 * n), 1u << 30);
                GC_TRY(pass("union_coo_sample", false, CooPart{COO_SAMPLE, every}, m / every + 32));
                GC_TRY(finalize_labels(v, s, s.P, st));
                return pass("union_coo", dense, CooPart{COO_REST, every}, m);
            }
            return pass("union_coo", dense, CooPart{COO_ALL, 0}, m);
        }
    });
}

}  // namespace gc
