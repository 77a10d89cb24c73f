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
//   m = 65,536 47 -> 36, 24 -> 25; m = 128,000 no gain.
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

// The COO finish of a static pass (every vertex a singleton at the start) has
// three forms: a union per thread (k_union_coo), one compared-and-queued pass over
// all edges (k_union_filter), and a sampled one: about 3n/4 to n edges, spread over
// the list, are united first (where a random graph's giant component appears),
// the trees are flattened, and the other edges then mostly find equal parents.
// Measured at 13 sizes of n from 12,000 to 2^22, m from n/2 to 16n, on ER, RMAT and
// grid + paths lists, by rule (m / n and microseconds: union per thread, chosen
// form).  The lines lie where neither kind of graph loses:
// - Fewer edges than the resident threads of 152 SMs (m < 49,152): comparing first
//   only adds a round trip (ER n = 32,768, m = n, Rem-CAS: 25 against 32).
// - 2^15 <= n <= 2^19: as many threads as vertices or more would start on singletons
//   at once and contend for the same few roots: sampled.  Rem with naive finds
//   from max(2n, 2^17) edges: ER n = 65,536 x 2 65, 44; x 16 101, 54; RMAT n = 2^18 x 8
//   139, 66; but n = 46,000 x 2 ER 60, 43 and RMAT 26, 35.  Union-Async with compressing
//   finds and Union-Hooks from 2n (n = 2^15 x 2: 81, 67; 86, 67).  Rules that shorten
//   their own walks (Early; split and halve) have less to gain: from max(2n, 2^18)
//   (Early, ER n = 2^18 x 4 69, 56; n = 92,000 x 2 32, 42), and Early with such a find
//   not at all (split, ER n = 131,072 x 8 81, 157; RMAT n = 2^18 x 8 167, 112).
//   Their second pass takes 8 rows of edges from 2^17 vertices and 4n edges (ER
//   n = 131,072 x 8, Early: 94 with 2 rows, 59 with 8), every other takes 2 (ER n = 2^15
//   x 4, Rem-CAS: 44; 44 with 2, 54 with 8).  Rules that compress nothing are sampled
//   at any n from 2^15: from 3n edges, from 2^18 vertices 2n (Union-Async, ER n = 65,536 x 2
//   63, 62, x 3 83, 63; n = 2^22 x 8 1,476, 503; Afforest, n = 65,536 x 2 30, 37).
// - n < 2^15: sampled from 8n edges (12,000 x 8: ER 55, 38, RMAT 25, 26), below one
//   pass (16,384 x 4: ER 55, 47, RMAT 23, 24); rules that shorten their own walks
//   sampled from 16n, else a union per thread, as are the rules that compress
//   nothing and Early with a compressing find.
// - n > 2^19: the first wave no longer covers the vertices; one pass from n edges
//   (n = 10^6 x 2: ER 182, 100, RMAT 76, 72; 2^22 x 1 257, 186).  Below, nearly every edge
//   links (n = 2^20 x 1/2: 40, 44; and at n <= 2^19 below 2n: grid + paths of 393,216
//   81, 104).  Rules that shorten their own walks up to 2^20 only from 8n (Early,
//   n = 10^6: ER x 8 147, 137, RMAT x 2 58, 77; n = 2^20: ER x 4 106, 121), and
//   Union-Async not there (split, RMAT n = 2^20 x 16 245, 289).
gconn_status union_coo_static(const Variant& v, const UFState& s, const uint32_t* edges, uint64_t m, cudaStream_t st) {
    if (v.link == GCONN_LINK_JTB || m < 49152) return union_coo(v, s, edges, m, 0, st);
    int L, F, S;
    uf_triple(v, &L, &F, &S);
    const int B = block_of(v);
    const uint64_t n = s.n;
    return dispatch_uf(L, F, S, s.sf != nullptr, [&]<int l, int f, int sp, bool sf>() -> gconn_status {
        if constexpr (l == LK_JTB) return GCONN_E_UNSUPPORTED;   // handled above
        else {
            auto pass = [&](const char* name, bool wide, CooPart part, uint64_t count) {
                auto k = wide ? k_union_filter<l, f, sp, sf, 8> : k_union_filter<l, f, sp, sf, 2>;
                return launch_pdl(name, k, grid_for(k, B, count / (wide ? 8 : 2) + 1), B, 0, st, (const uint2*)edges,
                                  m, s, part);
            };
            auto sampled = [&](bool wide) -> gconn_status {
                const uint32_t every = (uint32_t)std::min<uint64_t>(4 * m / (3 * n), 1u << 30);   // >= 2
                GC_TRY(pass("union_coo_sample", false, CooPart{COO_SAMPLE, every}, m / every + 32));
                GC_TRY(finalize_labels(v, s, s.P, st));
                return pass("union_coo", wide, CooPart{COO_REST, every}, m);
            };
            auto one_pass = [&](bool wide) { return pass("union_coo", wide, CooPart{COO_ALL, 0}, m); };
            auto per_thread = [&] { return union_coo(v, s, edges, m, 0, st); };

            constexpr bool hooks = l == LK_HOOKS, bare = rule_is_bare<l, f>();
            constexpr bool shortens = l == LK_EARLY || (!hooks && (f == FD_SPLIT || f == FD_HALVE));
            constexpr bool early_find = l == LK_EARLY && f != FD_NAIVE;
            if (n > (1u << 19) && !bare) {
                if (shortens && n <= (1u << 20))
                    return l != LK_ASYNC && m >= 8 * n ? one_pass(true) : per_thread();
                return m < n ? per_thread() : one_pass(m >= (shortens || l == LK_REMLOCK ? 4 : 2) * n);
            }
            if (bare && m < 2 * n) {
                if (hooks ? 2 * m >= 3 * n : l != LK_AFFOREST && n > (1u << 19) && m >= n) return one_pass(false);
                return per_thread();
            }
            if (early_find || (bare && n < (1u << 15))) return per_thread();
            if (n < (1u << 15)) {
                if (m >= (shortens ? 16 : 8) * n) return sampled(false);
                return shortens ? per_thread() : one_pass(false);
            }
            const uint64_t least = hooks || (l == LK_ASYNC && f == FD_COMPRESS) ? 2 * n
                                 : bare ? (n >= (1u << 18) ? 2 : 3) * n
                                 : std::max<uint64_t>(2 * n, 1u << (shortens ? 18 : 17));
            if (m < least) return per_thread();
            return sampled(shortens && n >= (1u << 17) && m >= 4 * n);
        }
    });
}

}  // namespace gc
