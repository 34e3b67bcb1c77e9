// Building blocks of the component kernels that keep a whole graph's rounds in
// one launch: edge passes of a gang of blocks (gang.cuh) over warp-private
// ranges, and active edges kept as pairs of roots.
#pragma once

#include "cc_device.cuh"
#include "common.cuh"
#include "gang.cuh"

namespace lrcc {

constexpr int GANG_EDGES = 4;                 // edges per lane and iteration
constexpr int GANG_STEP = 32 * GANG_EDGES;    // edges per warp and iteration

struct GangGraph {
    const int32_t* src;
    const int32_t* dst;
    int64_t m;
    int32_t n;
    int32_t* p;              // parents; the labels in the end
};

// Length of a warp's share of [0, total): whole iterations.
__host__ __device__ __forceinline__ int64_t gang_share(int64_t total, int64_t warps) {
    return ((total + warps - 1) / warps + GANG_STEP - 1) / GANG_STEP * GANG_STEP;
}
// This warp's share of [0, total), contiguous.
__device__ __forceinline__ void gang_range(const Gang& G, int64_t total, int64_t* lo, int64_t* hi) {
    const int64_t per = gang_share(total, G.warps());
    *lo = min(total, per * G.warp());
    *hi = min(total, *lo + per);
}

// GANG_EDGES edges per lane from [i, hi); ids outside [0, n) are reported and
// left out. VEC: src and dst are 16-byte aligned and i a multiple of 4.
template <bool VEC>
__device__ __forceinline__ void gang_load(const GangGraph& g, int64_t i, int64_t hi, uint64_t pol, int32_t (&u)[GANG_EDGES],
                                          int32_t (&v)[GANG_EDGES], bool (&ok)[GANG_EDGES], DevCtl* ctl) {
    const int lane = threadIdx.x & 31;
    if (VEC && i + GANG_STEP <= hi) {
        const int4 a = ld_stream_v4(g.src + i + lane * 4, pol);
        const int4 b = ld_stream_v4(g.dst + i + lane * 4, pol);
        u[0] = a.x; u[1] = a.y; u[2] = a.z; u[3] = a.w;
        v[0] = b.x; v[1] = b.y; v[2] = b.z; v[3] = b.w;
#pragma unroll
        for (int q = 0; q < GANG_EDGES; ++q) ok[q] = true;
    } else {
#pragma unroll
        for (int q = 0; q < GANG_EDGES; ++q) {
            const int64_t e = i + q * 32 + lane;
            ok[q] = e < hi;
            u[q] = ok[q] ? ld_stream(g.src + e, pol) : 0;
            v[q] = ok[q] ? ld_stream(g.dst + e, pol) : 0;
        }
    }
#pragma unroll
    for (int q = 0; q < GANG_EDGES; ++q)
        if (ok[q] && ((uint32_t)u[q] >= (uint32_t)g.n || (uint32_t)v[q] >= (uint32_t)g.n)) {
            record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)i);
            ok[q] = false;
            u[q] = v[q] = 0;
        }
}

// The edges a warp still has to join: pairs in a private stretch of the pair
// buffer, compacted in place, and, when more were kept than it holds, the rest
// of its two shares of the edge list (the sample, the edges after it), which is
// read again from iteration resume0 or resume1 on.
struct GangActive {
    static constexpr unsigned NONE = 0xFFFFFFFFu;
    int2* buf;               // this warp's stretch
    int cap;
    int count = 0;
    bool full = false;       // the current pass kept more than fits
    unsigned resume0 = NONE, resume1 = NONE;

    // Keeps the lanes' pairs of iteration `it` of share `part` (all lanes call
    // it); returns how many there were. Pairs are written only below what this
    // warp has already read.
    __device__ __forceinline__ int append(const bool (&keep)[GANG_EDGES], const int32_t (&a)[GANG_EDGES],
                                          const int32_t (&b)[GANG_EDGES], int part, unsigned it) {
        int cnt = 0;
#pragma unroll
        for (int q = 0; q < GANG_EDGES; ++q) cnt += keep[q];
        if (!__any_sync(0xffffffffu, cnt)) return 0;
        int total = 0;
        int at = count + warp_prefix_small(cnt, &total);
        if (full || count + total > cap) {
            full = true;
            if (part) resume1 = min(resume1, it);
            else resume0 = min(resume0, it);
        } else {
#pragma unroll
            for (int q = 0; q < GANG_EDGES; ++q)
                if (keep[q]) __stcs(buf + at++, make_int2(a[q], b[q]));
            count += total;
        }
        return total;
    }
};

// Roots of K vertices at once (x in, root out), by chase_step. Short chases
// store nothing: the pairs go on with the roots themselves, and with one large
// tree about, every lane would store to its old root's entry (57 us for 30,000
// such stores).
template <int K>
__device__ __forceinline__ void gang_roots(int32_t* p, int32_t (&x)[K], uint64_t keep) {
    int32_t v[K];
    unsigned live = (1u << K) - 1;
#pragma unroll
    for (int q = 0; q < K; ++q) v[q] = x[q];
    for (int step = 0; live; ++step) {
        int32_t nx[K];
#pragma unroll
        for (int q = 0; q < K; ++q)
            if (live >> q & 1) nx[q] = chase_step(p, v[q], x[q], step, keep);
#pragma unroll
        for (int q = 0; q < K; ++q)
            if (live >> q & 1) {
                if (nx[q] == x[q]) live &= ~(1u << q);
                x[q] = nx[q];
            }
    }
}

// Hooks the larger of two phase-start roots below the smaller, for the lanes
// with `on` (the whole warp calls it). Once a tree has grown large, most edges
// that leave it hook the same root, and atomics on one address run at about
// 1 G/s. So in the rounds (MATCH) the lanes that hook the same root send one atomic
// with the smallest of their ids (in passes over the edge list that costs more than
// it gains: 17.4 against 17.1 ms for 2048 graphs), and a block remembers the roots it hooks: slot -> (root,
// smallest id it was hooked below); an atomic that could not lower the parent
// any more is left out. That loses nothing: the earlier one is in p, and the
// edge is kept for the next pass like any other. Entries stay true from pass to
// pass, because a hooked root is never a root again. New roots enter a slot
// only on every sixteenth hook (`enter`), so that the many roots hooked once do
// not push out the few hooked all the time.
constexpr int HOOK_SLOTS = 1024;
template <bool MATCH>
__device__ __forceinline__ void gang_hook(int32_t* p, int32_t a, int32_t b, bool on, volatile uint64_t* s_hook,
                                          bool enter) {
    if (!__any_sync(0xffffffffu, on)) return;
    const int32_t hi = on ? max(a, b) : -1;
    int32_t lo = min(a, b);
    const unsigned same = MATCH ? __match_any_sync(0xffffffffu, hi) : 0u;
    if (!on) return;
    if (same & (same - 1)) lo = __reduce_min_sync(same, lo);
    if (same & lanemask_lt()) return;   // the first lane of each group goes on
    volatile uint64_t* slot = s_hook + (((uint32_t)hi * 0x9E3779B1u) >> 22);
    const uint64_t e = *slot;
    if (hi32(e) == (uint32_t)hi) {
        if ((int32_t)lo32(e) <= lo) return;
        enter = true;
    }
    if (enter || (same & (same - 1))) *slot = pack((uint32_t)lo, (uint32_t)hi);
    atomicMin(p + hi, lo);
}

// Joins the trees of a and b for good: only roots are linked (compare and
// swap) and only other entries are halved, so no link is replaced. For passes
// in which every link is made this way.
__device__ __forceinline__ void gang_join(int32_t* p, int32_t a, int32_t b, uint64_t keep) {
    for (;;) {
        a = find_root_halving(p, a, keep);
        b = find_root_halving(p, b, keep);
        if (a == b) return;
        const int32_t hi = max(a, b), lo = min(a, b);
        const int32_t old = atomicCAS(p + hi, hi, lo);
        if (old == hi) return;
        a = old;
        b = lo;
    }
}

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
// gathers need for their lines in flight (R-MAT scale 24, filter pass: 1.4 ms with
// 128 KB, 2.0 with 160 KB, 2.05 without a table).
enum Table { TABLE_NONE, TABLE_BITS, TABLE_TAGS };
constexpr int TABLE_BYTES = 130 << 10;
constexpr int64_t BITS_MAX_N = int64_t(TABLE_BYTES) * 8;
constexpr uint32_t TAG_SLOTS = TABLE_BYTES;
constexpr uint32_t TAG_NONE = 0x7F, TAG_MASK = 0x7F, TAG_KEEP = 0x80;
constexpr int64_t TAGS_MAX_N = int64_t(TAG_SLOTS) * TAG_NONE;

struct GangParams {
    GangGraph g;
    int64_t ms;              // sample: the first ms edges (ms = m: no sample)
    int64_t first;           // edges of the first pass
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

    // passes_ and edges_: those of the launches before this one
    __device__ __forceinline__ GangWork(const GangParams& P_, Gang& G_, DevCtl* c, volatile uint64_t* h, int passes_,
                                        unsigned long long edges_)
        : P(P_), G(G_), ctl(c), s_hook(h), stream_pol(policy_evict_first()), keep(policy_evict_last()),
          passes(passes_), edges(edges_) {
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
        gang_range(G, P.first, &lo, &hi);
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
        const unsigned warm = (unsigned)((hi - lo) / (12 * GANG_STEP));
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
                const bool clear = ((it / 16 + lane()) & 7) == 0;
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
                // learning costs as much as asking: in the first twelfth of the share, then
                // in every sixteenth iteration (1.98 -> 1.77 ms, R-MAT scale 24)
                if (it < warm || (it & 15) == 0)
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
                gang_hook<false>(p, a[q], b[q], ok[q], s_hook, enter(it));
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
    // every vertex to its root; false when the barrier gave up. When few pairs are left they are joined for good
    // in one pass.
    __device__ bool run_out(long long kept) {
        while (kept > 0) {
            if (passes >= P.max_passes) {
                if (lead()) record_error(ctl, LRCC_ERR_NOT_CONVERGED, passes);
                return true;
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
            if (kept < 0) return false;
        }
        shortcut<false>(0);
        return true;
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
__device__ __forceinline__ int32_t find_giant(const GangParams& P, int* s_key, int* s_cnt, unsigned long long* s_best, int* skewed,
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

}  // namespace lrcc
