// Connected components of one graph in one launch: the rounds of Sec. 4
// (Algorithm 4) inside a cooperative kernel, or, for a small graph, inside one
// block's shared memory.
//
// The rounds are those of cc.cu's hook rule 1 with two changes. An edge that
// still joins two trees is carried on as the pair of their roots, so after the
// first passes only roots are chased and a full shortcut over all vertices
// happens once at the end instead of once per round. And the pairs stay in
// stretches private to a warp, so nothing is appended through a shared counter
// and a round with few edges costs one barrier.
//
// Measured against the loop of launches (us): uniform 2^20 vertices, 2^22 edges
// 146 / 266; 1021 vertices, 2042 edges 17 / 56; paths of 8M vertices 383 / 926;
// R-MAT scale 20, 2^24 edges 144 / 2350; scale 24, 2^28 edges 2049 / 2498 (bound by
// the gathers the member table does not answer, one L2 request each).
//
// Why no connection is lost: a hook writes p[hi] = min(p[hi], lo) where hi was
// a root when this pass read it, and the edge that asked for it is kept as the
// pair (hi, lo). If another hook of the pass, or a chase storing its progress
// in p[hi], replaces that link, the kept pair still carries the connection into
// the next pass. A pair is dropped only when both ends reached one root. Links
// go from larger to smaller ids throughout, so no cycle forms, roots only ever
// become fewer, and in the end every root is the smallest id of its component.
#include <algorithm>
#include <cstddef>

#include "cc_gang.cuh"
#include "internal.h"

namespace lrcc {

namespace {

// ------------------------------------------------------------ one block

// Joins the trees of u and v in a shared-memory forest. Only roots are linked
// (compare and swap) and only other entries are halved, so no link is ever
// replaced and one call per edge labels the graph.
__device__ __forceinline__ void smem_join(volatile int* p, int u, int v) {
    auto root = [&](int x) {
        int px = p[x];
        while (px != x) {
            const int g = p[px];
            if (g != px) p[x] = g;
            x = px;
            px = g;
        }
        return x;
    };
    for (;;) {
        u = root(u);
        v = root(v);
        if (u == v) return;
        const int hi = max(u, v), lo = min(u, v);
        const int old = atomicCAS(const_cast<int*>(p) + hi, hi, lo);
        if (old == hi) return;
        u = old;
        v = lo;
    }
}

__global__ void __launch_bounds__(GANG_THREADS, 1)
    cc_one_block(const int32_t* __restrict__ src, const int32_t* __restrict__ dst, int m, int n,
                 int32_t* __restrict__ label, DevCtl* ctl) {
    extern __shared__ int one_p[];
    volatile int* p = one_p;
    for (int v = threadIdx.x; v < n; v += GANG_THREADS) p[v] = v;
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += 4 * GANG_THREADS) {
        int u[4], v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int e = i + q * GANG_THREADS;
            u[q] = e < m ? __ldg(src + e) : 0;
            v[q] = e < m ? __ldg(dst + e) : 0;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if ((uint32_t)u[q] >= (uint32_t)n || (uint32_t)v[q] >= (uint32_t)n)
                record_error(ctl, LRCC_ERR_INVALID_INPUT, i + q * GANG_THREADS);
            else
                smem_join(p, u[q], v[q]);
        }
    }
    __syncthreads();
    for (int v = threadIdx.x; v < n; v += GANG_THREADS) {
        int x = p[v];
        for (int y; (y = p[x]) != x;) x = y;
        label[v] = x;
    }
    if (threadIdx.x == 0) {
        ctl->rounds = 1;
        ctl->edges_read = (unsigned long long)m;
    }
}

// ------------------------------------------------------------ the gang

// Membership table of the giant tree, in shared memory while the edges after
// the sample are filtered: an edge with both ends in it needs no read of p.
//   BITS  one bit per vertex, for graphs it holds.
//   TAGS  a direct-mapped cache of members met so far, one byte per slot: vertex
//         v has slot v mod TAG_SLOTS and tag v / TAG_SLOTS. A tag that was hit is
//         protected; another member takes a protected slot only after one in
//         eight of its misses has cleared the mark, so that a slot stays with
//         its most frequent vertices. Membership never ends (trees only merge),
//         so an entry is never wrong. A warp whose vertices hit less than one
//         time in 32 stops asking.
// 130 KB is the best size on GB300: the rest of the 256 KB is L1, which the
// gathers need for their lines in flight (R-MAT scale 24, filter pass: 1.43 ms
// with 128 KB, 2.0 with 160 KB, 2.05 without a table).
enum Table { TABLE_NONE, TABLE_BITS, TABLE_TAGS };
constexpr int TABLE_BYTES = 130 << 10;
constexpr int64_t BITS_MAX_N = int64_t(TABLE_BYTES) * 8;
constexpr uint32_t TAG_SLOTS = TABLE_BYTES;
constexpr uint32_t TAG_NONE = 0x7F, TAG_MASK = 0x7F, TAG_KEEP = 0x80;
constexpr int64_t TAGS_MAX_N = int64_t(TAG_SLOTS) * TAG_NONE;

struct GangParams {
    GangGraph g;
    int64_t ms;              // sample: the first ms edges (ms = m: no sample)
    int sample_passes;       // passes over the sample before the other edges are filtered
    bool first_min;          // first pass: link endpoints without reading their parents
    int2* buf;               // capw pairs per warp
    int capw;
    int2* left;              // per warp: what the sample's passes left (pairs, resume0)
    int32_t* giant;          // the giant's root, and whether a few vertices have most of the edges
    int only;                // filter: run when giant[1] has this value (-1: always)
    uint32_t* bits;          // TABLE_BITS: membership, one bit per vertex
    int max_passes;
    int64_t join;            // at most this many pairs left: join them for good in one pass
};

// Root of v, reading only.
__device__ __forceinline__ int32_t root_of(const int32_t* p, int32_t v, uint64_t keep) {
    for (;;) {
        const int32_t x = ld_hint(p + v, keep);
        if (x == v) return v;
        v = x;
    }
}

// One block's view of the gang's work on one graph.
template <bool VEC>
struct GangWork {
    const GangParams& P;
    Gang& G;
    DevCtl* ctl;
    volatile uint64_t* s_hook;   // HOOK_SLOTS entries (gang_hook)
    uint64_t stream_pol, keep;
    GangActive act;
    int passes;                  // passes so far (before this launch included)
    unsigned long long edges;    // edges read so far

    __device__ __forceinline__ GangWork(const GangParams& P_, Gang& G_, DevCtl* c, volatile uint64_t* h)
        : P(P_), G(G_), ctl(c), s_hook(h), stream_pol(policy_evict_first()), keep(policy_evict_last()),
          passes(c->rounds), edges(c->edges_read) {
        act.buf = P.buf + (int64_t)G.warp() * P.capw;
        act.cap = P.capw;
    }
    __device__ __forceinline__ static int lane() { return threadIdx.x & 31; }
    __device__ __forceinline__ bool lead() const { return G.rank == 0 && threadIdx.x == 0; }
    // every sixteenth hook of a lane may enter its root into s_hook
    __device__ __forceinline__ static bool enter(unsigned it) { return ((it + lane()) & 15) == 0; }

    // Every vertex of this warp's share to its root. BITS: also the giant's bit map.
    template <bool BITS>
    __device__ void shortcut(int32_t giant) {
        int32_t* p = P.g.p;
        int64_t lo, hi;
        gang_range(G, P.g.n, &lo, &hi);
        for (int64_t i = lo; i < hi; i += GANG_STEP) {
            int32_t x[GANG_EDGES], old[GANG_EDGES];
            unsigned live = 0;
#pragma unroll
            for (int q = 0; q < GANG_EDGES; ++q) {
                const int64_t v = i + q * 32 + lane();
                old[q] = x[q] = v < hi ? ld_cg(p + v) : -1;
                if (v < hi && x[q] != (int32_t)v) live |= 1u << q;
            }
            for (int step = 0; live; ++step) {
                int32_t nx[GANG_EDGES];
#pragma unroll
                for (int q = 0; q < GANG_EDGES; ++q)
                    if (live >> q & 1) nx[q] = chase_step(p, (int32_t)(i + q * 32 + lane()), x[q], step, keep);
#pragma unroll
                for (int q = 0; q < GANG_EDGES; ++q)
                    if (live >> q & 1) {
                        if (nx[q] == x[q]) live &= ~(1u << q);
                        x[q] = nx[q];
                    }
            }
#pragma unroll
            for (int q = 0; q < GANG_EDGES; ++q) {
                const int64_t v = i + q * 32 + lane();
                if (v < hi && x[q] != old[q]) p[v] = x[q];
                if (BITS) {
                    const unsigned w = __ballot_sync(0xffffffffu, v < hi && x[q] == giant);
                    if (lane() == 0 && i + q * 32 < hi) P.bits[(i >> 5) + q] = w;
                }
            }
        }
    }

    // First pass over the sample: every parent is the vertex itself. Either
    // both parents are read and the larger hooked below the smaller (edges met
    // later then hook what earlier ones linked to: best when the pass is long
    // against the edges in flight), or the endpoints themselves are linked, one
    // atomic per edge and no read. Links may replace one another: all these
    // edges are read again.
    __device__ void first_pass() {
        int32_t u[GANG_EDGES], v[GANG_EDGES];
        bool ok[GANG_EDGES];
        int64_t lo, hi;
        gang_range(G, P.ms, &lo, &hi);
        unsigned it = 0;
        for (int64_t i = lo; i < hi; i += GANG_STEP, ++it) {
            gang_load<VEC>(P.g, i, hi, stream_pol, u, v, ok, ctl);
            if (!P.first_min) {
                int32_t a[GANG_EDGES], b[GANG_EDGES];
#pragma unroll
                for (int q = 0; q < GANG_EDGES; ++q) {
                    a[q] = ld_hint(P.g.p + u[q], keep);
                    b[q] = ld_hint(P.g.p + v[q], keep);
                }
#pragma unroll
                for (int q = 0; q < GANG_EDGES; ++q) {
                    u[q] = a[q];
                    v[q] = b[q];
                }
            }
#pragma unroll
            for (int q = 0; q < GANG_EDGES; ++q)
                gang_hook<false>(P.g.p, u[q], v[q], ok[q] && u[q] != v[q], s_hook, enter(it));
        }
        ++passes;
        edges += (unsigned long long)P.ms;
    }

    // This warp's share of the sample (part 0) or of the edges after it (part 1).
    __device__ __forceinline__ void share(int part, int64_t* lo, int64_t* hi) const {
        gang_range(G, part ? P.g.m - P.ms : P.ms, lo, hi);
        if (part) {
            *lo += P.ms;
            *hi += P.ms;
        }
    }

    // A pass over one share of the edge list while every tree is a star; the
    // table answers for members of the giant. Returns how many edges this warp kept.
    template <int TABLE>
    __device__ int star_pass(int part, int32_t giant, unsigned char* s_table) {
        int32_t* p = P.g.p;
        int64_t lo, hi;
        share(part, &lo, &hi);
        int kept = 0;
        unsigned it = 0;
        int32_t u[GANG_EDGES], v[GANG_EDGES];
        bool ok[GANG_EDGES];
        bool ask = TABLE != TABLE_NONE;
        int hits = 0;
        for (int64_t i = lo; i < hi; i += GANG_STEP, ++it) {
            gang_load<VEC>(P.g, i, hi, stream_pol, u, v, ok, ctl);
            int32_t a[GANG_EDGES], b[GANG_EDGES];
            if (TABLE == TABLE_NONE || !ask) {
#pragma unroll
                for (int q = 0; q < GANG_EDGES; ++q) {
                    a[q] = ld_hint(p + u[q], keep);
                    b[q] = ld_hint(p + v[q], keep);
                }
            } else if (TABLE == TABLE_BITS) {
                const uint32_t* bits = reinterpret_cast<const uint32_t*>(s_table);
#pragma unroll
                for (int q = 0; q < GANG_EDGES; ++q) {
                    const bool in_u = bits[u[q] >> 5] >> (u[q] & 31) & 1;
                    const bool in_v = bits[v[q] >> 5] >> (v[q] & 31) & 1;
                    a[q] = b[q] = giant;
                    if (!in_u) a[q] = ld_cg_hint(p + u[q], keep);
                    if (!in_v) b[q] = ld_cg_hint(p + v[q], keep);
                }
            } else {
                uint32_t eu[GANG_EDGES], ev[GANG_EDGES];
#pragma unroll
                for (int q = 0; q < GANG_EDGES; ++q) {
                    eu[q] = s_table[(uint32_t)u[q] % TAG_SLOTS];
                    ev[q] = s_table[(uint32_t)v[q] % TAG_SLOTS];
                    const bool in_u = (eu[q] & TAG_MASK) == (uint32_t)u[q] / TAG_SLOTS;
                    const bool in_v = (ev[q] & TAG_MASK) == (uint32_t)v[q] / TAG_SLOTS;
                    hits += in_u + in_v;
                    a[q] = b[q] = giant;
                    // straight from L2: with the table L1 is small, and its lines are
                    // better spent on reads in flight (1.60 -> 1.43 ms)
                    if (!in_u) a[q] = ld_cg_hint(p + u[q], keep);
                    if (!in_v) b[q] = ld_cg_hint(p + v[q], keep);
                }
                const bool clear = ((it + lane()) & 7) == 0;
                auto learn = [&](int32_t x, uint32_t e, int32_t root) {
                    const uint32_t tag = (uint32_t)x / TAG_SLOTS;
                    unsigned char* slot = s_table + (uint32_t)x % TAG_SLOTS;
                    if ((e & TAG_MASK) == tag) {
                        if (!(e & TAG_KEEP)) *slot = (unsigned char)(tag | TAG_KEEP);
                    } else if (root == giant) {
                        if (!(e & TAG_KEEP)) *slot = (unsigned char)tag;
                        else if (clear) *slot = (unsigned char)(e & TAG_MASK);
                    }
                };
#pragma unroll
                for (int q = 0; q < GANG_EDGES; ++q)
                    if (ok[q]) {
                        learn(u[q], eu[q], a[q]);
                        learn(v[q], ev[q], b[q]);
                    }
                if ((it & 31) == 31) {
                    // 32 iterations of 8 lookups per lane
                    if (__reduce_add_sync(0xffffffffu, hits) < 32 * 8) ask = false;
                    hits = 0;
                }
            }
#pragma unroll
            for (int q = 0; q < GANG_EDGES; ++q) {
                ok[q] = ok[q] && a[q] != b[q];
                gang_hook<true>(p, a[q], b[q], ok[q], s_hook, enter(it));
            }
            kept += act.append(ok, a, b, part, it);
        }
        return kept;
    }

    // Calls f(u, v, ok, part, it) for the pairs this warp carries and for the
    // edges that did not fit; act is empty before the first call.
    template <class F>
    __device__ void each_pair(F f) {
        int32_t u[GANG_EDGES], v[GANG_EDGES];
        bool ok[GANG_EDGES];
        const int count = act.count;
        const unsigned from0 = act.resume0, from1 = act.resume1;
        act.count = 0;
        act.full = false;
        act.resume0 = act.resume1 = GangActive::NONE;
        unsigned it = 0;
        for (int i = 0; i < count; i += GANG_STEP, ++it) {
#pragma unroll
            for (int q = 0; q < GANG_EDGES; ++q) {
                const int e = i + q * 32 + lane();
                ok[q] = e < count;
                const int2 x = ok[q] ? __ldcs(act.buf + e) : make_int2(0, 0);
                u[q] = x.x;
                v[q] = x.y;
            }
            f(u, v, ok, 0, it);   // compaction in place always fits
        }
#pragma unroll 1
        for (int part = 0; part < 2; ++part) {
            it = part ? from1 : from0;
            if (it == GangActive::NONE) continue;
            int64_t lo, hi;
            share(part, &lo, &hi);
            for (int64_t i = lo + (int64_t)it * GANG_STEP; i < hi; i += GANG_STEP, ++it) {
                gang_load<VEC>(P.g, i, hi, stream_pol, u, v, ok, ctl);
                f(u, v, ok, part, it);
            }
        }
    }

    // One round: the carried pairs to their roots, hooked and kept while the
    // roots differ. Returns how many this warp kept.
    __device__ int round() {
        int kept = 0;
        each_pair([&](int32_t(&u)[GANG_EDGES], int32_t(&v)[GANG_EDGES], bool(&ok)[GANG_EDGES], int part, unsigned it) {
            // two edges at a time: eight chases at once need more registers than there are
#pragma unroll
            for (int h = 0; h < GANG_EDGES; h += 2) {
                int32_t x[4] = {u[h], v[h], u[h + 1], v[h + 1]};
                gang_roots(P.g.p, x, keep);
                u[h] = x[0];
                v[h] = x[1];
                u[h + 1] = x[2];
                v[h + 1] = x[3];
            }
#pragma unroll
            for (int q = 0; q < GANG_EDGES; ++q) {
                ok[q] = ok[q] && u[q] != v[q];
                gang_hook<true>(P.g.p, u[q], v[q], ok[q], s_hook, enter(it));
            }
            kept += act.append(ok, u, v, part, it);
        });
        return kept;
    }

    // Ends a pass: how many pairs the gang kept (the counters take turns), or -1
    // when the barrier gave up.
    __device__ long long settle(int kept) {
        if (lane() == 0 && kept) atomicAdd(&G.g->kept[passes % 3], (unsigned long long)kept);
        if (lead()) G.g->kept[(passes + 1) % 3] = 0;
        if (!G.sync()) return -1;
        const long long total = (long long)*reinterpret_cast<volatile unsigned long long*>(&G.g->kept[passes % 3]);
        ++passes;
        return total;
    }

    // Rounds until nothing is left to join (`kept` pairs to begin with), then
    // every vertex to its root. When few pairs are left they are joined for good
    // in one pass.
    __device__ void run_out(long long kept) {
        while (kept > 0) {
            if (passes >= P.max_passes) {
                if (lead()) record_error(ctl, LRCC_ERR_NOT_CONVERGED, passes);
                return report();
            }
            edges += (unsigned long long)kept;
            if (kept <= P.join) {
                each_pair([&](int32_t(&u)[GANG_EDGES], int32_t(&v)[GANG_EDGES], bool(&ok)[GANG_EDGES], int, unsigned) {
#pragma unroll 1
                    for (int q = 0; q < GANG_EDGES; ++q)
                        if (ok[q]) gang_join(P.g.p, u[q], v[q], keep);
                });
                kept = settle(0);
            } else {
                kept = settle(round());
            }
            if (kept < 0) return;
        }
        shortcut<false>(0);
        report();
    }
    __device__ void report() {
        if (lead()) {
            ctl->rounds = passes;
            ctl->edges_read = edges;
        }
    }
};

// The tree most sampled edge ends belong to (every block computes the same one),
// and whether the sample meets a few vertices again and again: of 1024 edge ends
// of an R-MAT graph of scale 24 about ten pairs name the same vertex, of a
// uniform graph of that size hardly ever one.
__device__ int32_t find_giant(const GangParams& P, int* s_key, int* s_cnt, unsigned long long* s_best, int* skewed,
                              uint64_t keep) {
    constexpr int SLOTS = 2 * GANG_THREADS;
    const int64_t e = (int64_t)(((uint64_t)mix32(threadIdx.x + 1) * (uint64_t)P.ms) >> 32);
    const int32_t v = __ldg(P.g.src + e);
    const bool in = (uint32_t)v < (uint32_t)P.g.n;
    // counts the threads' keys by value in an open table (at most GANG_THREADS
    // keys in twice as many slots); returns how many came before this one
    auto tally = [&](int32_t key) {
        for (int t = threadIdx.x; t < SLOTS; t += GANG_THREADS) {
            s_key[t] = -1;
            s_cnt[t] = 0;
        }
        __syncthreads();
        int before = 0;
        if (in) {
            int s = (int)(mix32((uint32_t)key) & (SLOTS - 1));
            for (;;) {
                const int k = atomicCAS(&s_key[s], -1, key);
                if (k == -1 || k == key) break;
                s = (s + 1) & (SLOTS - 1);
            }
            before = atomicAdd(&s_cnt[s], 1);
        }
        __syncthreads();
        return before;
    };
    *skewed = __syncthreads_count(tally(v) > 0) >= 3;
    tally(in ? root_of(P.g.p, v, keep) : 0);
    if (threadIdx.x == 0) *s_best = 0;
    __syncthreads();
    for (int t = threadIdx.x; t < SLOTS; t += GANG_THREADS)
        if (s_cnt[t]) atomicMax(s_best, ((unsigned long long)s_cnt[t] << 32) | (uint32_t)~s_key[t]);
    __syncthreads();
    return *s_best ? (int32_t)~(uint32_t)*s_best : 0;
}

// The whole labelling, or, with a sample, its passes over the sample.
template <bool VEC, bool BITS>
__global__ void __launch_bounds__(GANG_THREADS, 1) cc_gang_kernel(const __grid_constant__ GangParams P, GangCtl* gc, DevCtl* ctl) {
    __shared__ int s_flag;
    __shared__ uint64_t s_hook[HOOK_SLOTS];
    __shared__ int s_key[2 * GANG_THREADS], s_cnt[2 * GANG_THREADS];
    __shared__ unsigned long long s_best;
    static_assert(HOOK_SLOTS == GANG_THREADS, "one slot per thread");
    s_hook[threadIdx.x] = ~0ull;
    Gang G{gc, &gc->arrived[0], (int)gridDim.x, (int)blockIdx.x, 0, ctl, &s_flag};
    GangWork<VEC> w(P, G, ctl, s_hook);
    for (int64_t v = (int64_t)blockIdx.x * GANG_THREADS + threadIdx.x; v < P.g.n; v += (int64_t)gridDim.x * GANG_THREADS)
        P.g.p[v] = (int32_t)v;
    if (!G.sync()) return;
    w.first_pass();
    if (!G.sync()) return;
    long long kept = 0;
    const bool sampled = P.ms < P.g.m;
    if (!sampled || P.sample_passes > 1) {
        w.template shortcut<false>(0);
        if (!G.sync()) return;
        w.edges += (unsigned long long)P.ms;
        kept = w.settle(w.template star_pass<TABLE_NONE>(0, 0, nullptr));
        if (kept < 0) return;
    }
    if (!sampled) {
        if (kept == 0) return w.report();   // the trees were stars and none was joined
        return w.run_out(kept);
    }
    for (int r = 2; r < P.sample_passes && kept > 0; ++r) {
        w.edges += (unsigned long long)kept;
        kept = w.settle(w.round());
        if (kept < 0) return;
    }
    int skewed;
    const int32_t giant = find_giant(P, s_key, s_cnt, &s_best, &skewed, w.keep);
    w.template shortcut<BITS>(giant);
    if (w.lane() == 0) P.left[G.warp()] = make_int2(w.act.count, (int)w.act.resume0);
    if (w.lead()) {
        P.giant[0] = giant;
        P.giant[1] = skewed;
    }
    w.report();
}

// The edges after the sample (all edges when the sample was passed over only
// once), and the rounds that are left.
template <bool VEC, int TABLE>
__global__ void __launch_bounds__(GANG_THREADS, 1) cc_filter_kernel(const __grid_constant__ GangParams P, GangCtl* gc, DevCtl* ctl) {
    extern __shared__ __align__(16) unsigned char s_table[];
    __shared__ int s_flag;
    __shared__ uint64_t s_hook[HOOK_SLOTS];
    if (ctl->status == LRCC_ERR_TIMEOUT || (P.only >= 0 && P.giant[1] != P.only)) return;
    s_hook[threadIdx.x] = ~0ull;
    Gang G{gc, &gc->arrived[1], (int)gridDim.x, (int)blockIdx.x, 0, ctl, &s_flag};
    GangWork<VEC> w(P, G, ctl, s_hook);
    const int32_t giant = *P.giant;
    const bool again = P.sample_passes == 1;   // the sample's edges were not kept
    int kept_warp = 0;
    if (!again) {
        const int2 left = P.left[G.warp()];
        w.act.count = left.x;
        w.act.resume0 = (unsigned)left.y;
        w.act.full = w.act.resume0 != GangActive::NONE;
        kept_warp = left.x + (w.act.full ? 1 : 0);
    }
    if (TABLE == TABLE_BITS)
        for (int i = threadIdx.x; i < (int)((P.g.n + 31) >> 5); i += GANG_THREADS)
            reinterpret_cast<uint32_t*>(s_table)[i] = __ldcg(P.bits + i);
    if (TABLE == TABLE_TAGS)
        for (int i = threadIdx.x; i < TABLE_BYTES / 4; i += GANG_THREADS)
            reinterpret_cast<uint32_t*>(s_table)[i] = TAG_NONE * 0x01010101u;
    __syncthreads();
    // the sample's share (when it was not kept) and the share of the edges after it
#pragma unroll 1
    for (int part = again ? 0 : 1; part < 2; ++part) kept_warp += w.template star_pass<TABLE>(part, giant, s_table);
    w.edges += (unsigned long long)(P.g.m - (again ? 0 : P.ms));
    const long long kept = w.settle(kept_warp);
    if (kept < 0) return;
    if (kept == 0) return w.report();
    w.run_out(kept);
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// The one-block kernel's limits: its forest in shared memory, and as many
// edges as one SM joins in the time the gang's barriers take.
constexpr int64_t ONE_MAX_N = 48 << 10;
constexpr int64_t ONE_MAX_M = 24 << 10;

struct GangShape {
    int blocks, capw;
    size_t off_left, off_bits, bytes;   // behind the pairs: what each warp left, the giant, the bit map
};

GangShape gang_shape(int64_t m, int64_t n, int sms) {
    GangShape s;
    // a block for every 2048 edges or vertices: small graphs have cheaper barriers
    s.blocks = (int)std::max<int64_t>(1, std::min<int64_t>(sms, (std::max(m, n) + 2047) / 2048));
    const int64_t warps = (int64_t)s.blocks * GANG_WARPS;
    // Pairs for three eighths of the edges (paths keep a third of theirs after
    // the first passes), for a quarter above 2^26 edges; a warp that keeps more
    // reads the rest of its share again. Only the warps that have a share count.
    const int64_t per = gang_share(m, warps);
    s.capw = (int)(m <= (int64_t(1) << 26) ? per * 3 / 8 : per / 4) + 16;
    const int64_t used = std::min(warps, (m + GANG_STEP - 1) / GANG_STEP);   // the sample's shares are shorter
    s.off_left = align_up(sizeof(int2) * (size_t)s.capw * (size_t)std::max<int64_t>(used, 1), 256);
    s.off_bits = s.off_left + align_up(sizeof(int2) * (size_t)(warps + 1), 256);
    s.bytes = s.off_bits + (n <= BITS_MAX_N ? align_up((size_t)(n + 31) / 32 * 4, 256) : 0);
    return s;
}

lrcc_status launch_gang(Ctx* c, const void* kernel, GangParams& P, int blocks, size_t smem) {
    if (smem) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    GangCtl* gc = reinterpret_cast<GangCtl*>(reinterpret_cast<char*>(c->ctl) + offsetof(DevCtl, gang));
    DevCtl* ctl = c->ctl;
    void* args[] = {&P, &gc, &ctl};
    return cuda_status(cudaLaunchCooperativeKernel(kernel, dim3(blocks), dim3(GANG_THREADS), args, smem, c->stream));
}

}  // namespace

bool cc_gang_applies(const Plan& p) { return p.cc_hook == 1 && p.cc_max_rounds == 0 && p.use_graphs != 2; }

bool cc_one_block_applies(int64_t m, int64_t n) { return n <= ONE_MAX_N && m <= ONE_MAX_M; }

size_t cc_gang_ws(int64_t m, int64_t n, int sms) {
    return cc_one_block_applies(m, n) ? 0 : gang_shape(m, n, sms).bytes;
}

lrcc_status cc_run_gang(Ctx* c, const int32_t* src, const int32_t* dst, int64_t m, int64_t n, int32_t* label,
                        const Plan& p) {
    if (cc_one_block_applies(m, n)) {
        const size_t smem = sizeof(int) * (size_t)n;
        cudaFuncSetAttribute((const void*)cc_one_block, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        phase_begin(c, c->stream);
        cc_one_block<<<1, GANG_THREADS, smem, c->stream>>>(src, dst, (int)m, (int)n, label, c->ctl);
        phase_end(c, c->stream, PH_CC_LOOP);
        return cuda_status(cudaGetLastError());
    }
    const GangShape S = gang_shape(m, n, c->sms);
    char* ws = static_cast<char*>(c->ws);
    GangParams P;
    P.g = GangGraph{src, dst, m, (int32_t)n, label};
    P.buf = reinterpret_cast<int2*>(ws);
    P.capw = S.capw;
    P.left = reinterpret_cast<int2*>(ws + S.off_left);
    P.giant = reinterpret_cast<int32_t*>(P.left + S.blocks * GANG_WARPS);
    P.only = -1;
    P.bits = reinterpret_cast<uint32_t*>(ws + S.off_bits);
    int lg = 0;
    while ((int64_t(1) << lg) < n) ++lg;
    P.max_passes = 64 + 4 * lg;
    // Few pairs left over: join them for good, where no tree is expected to hold
    // most of the graph (forests: paths of 8M vertices 381 us against 426 without).
    // With a giant tree the joins contend for its root: uniform graphs of 2^17
    // vertices and edges 96 us against 56.
    P.join = m < n ? std::min(int64_t(1) << 18, n / 8) : 0;
    // The sample: the first m / k edges (plan.cc_sample = k). Automatically one
    // edge per vertex from 2 edges per vertex up: a random graph's giant tree
    // then holds most vertices, and the edges after the sample are mostly
    // dropped unread of their roots (2^20 vertices, 4 edges each: 142 us, 246
    // without). Below 2^19 edges a second launch costs what it saves (R-MAT scale
    // 14: 42 us without a sample, 57 with); with 1.5 edges per vertex half the
    // edges pay from 2^22 vertices on (2^24: 1111 against 1268 us; 2^20: 139
    // against 128).
    int64_t ms = m;
    if (p.cc_sample > 1) ms = m / p.cc_sample;
    else if (p.cc_sample < 0 && m >= (int64_t(1) << 19))
        ms = m >= 2 * n ? n : n >= (int64_t(1) << 22) && 2 * m >= 3 * n ? m / 2 : m;
    P.ms = ms >= 4096 ? ms & ~int64_t(3) : m;
    const bool sampled = P.ms < m;
    // Long passes over dense graphs: one pass that reads the parents forms the
    // giant (edges met later hook to what earlier ones made). In short ones most
    // edges are in flight at once, and three passes are needed (R-MAT scale 18: 83
    // us against 160), the first of which need not read the parents unless the
    // pass is long or the graph dense.
    P.sample_passes = m >= 8 * n && P.ms >= (int64_t(1) << 20) ? 1 : 3;
    P.first_min = sampled ? P.sample_passes > 1 && P.ms < (int64_t(1) << 22) : m < 2 * n;
    const int table = !sampled ? TABLE_NONE : n <= BITS_MAX_N ? TABLE_BITS : n <= TAGS_MAX_N ? TABLE_TAGS : TABLE_NONE;
    const bool vec = aligned16(src) && aligned16(dst);
    const bool bits = table == TABLE_BITS;
    phase_begin(c, c->stream);
    lrcc_status st = launch_gang(c,
                                 vec ? (bits ? (const void*)cc_gang_kernel<true, true> : (const void*)cc_gang_kernel<true, false>)
                                     : (bits ? (const void*)cc_gang_kernel<false, true> : (const void*)cc_gang_kernel<false, false>),
                                 P, S.blocks, 0);
    auto filter = [&](int t, int only) {
        const void* k = t == TABLE_BITS ? (vec ? (const void*)cc_filter_kernel<true, TABLE_BITS>
                                               : (const void*)cc_filter_kernel<false, TABLE_BITS>)
                      : t == TABLE_TAGS ? (vec ? (const void*)cc_filter_kernel<true, TABLE_TAGS>
                                               : (const void*)cc_filter_kernel<false, TABLE_TAGS>)
                                        : (vec ? (const void*)cc_filter_kernel<true, TABLE_NONE>
                                               : (const void*)cc_filter_kernel<false, TABLE_NONE>);
        P.only = only;
        st = launch_gang(c, k, P, S.blocks, t == TABLE_NONE ? 0 : TABLE_BYTES);
    };
    if (st == LRCC_OK && sampled) {
        // the cache of members pays when a few vertices have most of the edges,
        // which the sample tells on the device: the other kernel returns at once
        filter(table, table == TABLE_TAGS ? 1 : -1);
        if (st == LRCC_OK && table == TABLE_TAGS) filter(TABLE_NONE, 0);
    }
    phase_end(c, c->stream, PH_CC_LOOP);
    return st;
}

}  // namespace lrcc
