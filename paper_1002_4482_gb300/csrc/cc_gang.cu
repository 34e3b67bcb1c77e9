// Connected components of one graph in one launch: the rounds of Sec. 4
// (Algorithm 4) inside a cooperative kernel, or, for a small graph, inside one
// block's shared memory.
//
// The rounds are those of cc.cu's hook rule 1 with two changes. An edge that
// still joins two trees is carried on as the pair of their roots, so after the
// first passes only roots are chased and a full shortcut over all vertices
// happens once at the end instead of once per round. And the pairs stay in
// stretches private to a warp, so nothing is appended through a shared counter
// and a round with few edges costs one barrier. Labelling a part of the edges
// first and leaving out what lies inside the largest tree after it is the idea of
// Afforest (Sutton, Ben-Nun, Barak, "Optimizing Parallel Graph Connectivity
// Computation via Subgraph Sampling", IPDPS 2018).
//
// Measured against the loop of launches (us): uniform 2^20 vertices, 2^22 edges
// 146 / 266; 1021 vertices, 2042 edges 11-15 / 50-56; paths of 8M vertices 383 / 926;
// R-MAT scale 20, 2^24 edges 144 / 2350; scale 24, 2^28 edges 1725 / 2498 (bound by
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
        clear_stats(ctl);   // a call of one launch has no memset before it
        ctl->rounds = 1;
        ctl->edges_read = (unsigned long long)m;
    }
}

// ------------------------------------------------------------ the gang

// The whole labelling, or, with a sample, its passes over the sample.
template <bool VEC, bool BITS>
__global__ void __launch_bounds__(GANG_THREADS, 1) cc_gang_kernel(const __grid_constant__ GangParams P, GangCtl* gc, DevCtl* ctl) {
    __shared__ int s_flag;
    __shared__ uint64_t s_hook[HOOK_SLOTS];
    __shared__ int s_key[2 * GANG_THREADS], s_cnt[2 * GANG_THREADS];
    __shared__ unsigned long long s_best;
    for (int h = threadIdx.x; h < HOOK_SLOTS; h += GANG_THREADS) s_hook[h] = ~0ull;
    Gang G{gc, &gc->arrived[0], (int)gridDim.x, (int)blockIdx.x, 0, ctl, &s_flag};
    GangWork<VEC> w(P, G, ctl, s_hook, ctl->rounds, ctl->edges_read);
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
        // (with nothing kept the trees were stars and none was joined)
        if (kept > 0 && !w.run_out(kept)) return;
        return w.report();
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
    // gave_up first: the sample's launch has then written neither P.giant nor P.left
    if (ctl->gave_up || (P.only >= 0 && P.giant[1] != P.only)) return;
    for (int h = threadIdx.x; h < HOOK_SLOTS; h += GANG_THREADS) s_hook[h] = ~0ull;
    Gang G{gc, &gc->arrived[1], (int)gridDim.x, (int)blockIdx.x, 0, ctl, &s_flag};
    GangWork<VEC> w(P, G, ctl, s_hook, ctl->rounds, ctl->edges_read);
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
    if (kept > 0 && !w.run_out(kept)) return;
    w.report();
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

GangShape gang_shape(int64_t m, int64_t n, int sms, bool tight) {
    GangShape s;
    // a block for every 2048 edges or vertices: small graphs have cheaper barriers
    s.blocks = (int)std::max<int64_t>(1, std::min<int64_t>(sms, (std::max(m, n) + 2047) / 2048));
    const int64_t warps = (int64_t)s.blocks * GANG_WARPS;
    // Pairs for three quarters of the edges of a sparse graph (a uniform one of 1
    // edge per vertex keeps two thirds after the first passes: 104 us, 128 with
    // half the room), for three eighths where a sample leaves fewer, for a quarter
    // above 2^26 edges; a warp that keeps more reads the rest of its share again, so a
    // quarter will do where memory is accounted for (tight). Only the warps that have a
    // share count.
    const int64_t per = gang_share(m, warps);
    s.capw = (int)(tight || m > (int64_t(1) << 26) ? per / 4 : m < 2 * n ? per * 3 / 4 : per * 3 / 8) + 16;
    s.capw = std::max(s.capw, GANG_STEP);   // one iteration's pairs, also of a short sample
    const int64_t used = std::min(warps, (m + GANG_STEP - 1) / GANG_STEP);   // the sample's shares are shorter
    s.off_left = align_up(sizeof(int2) * (size_t)s.capw * (size_t)std::max<int64_t>(used, 1), 256);
    s.off_bits = s.off_left + align_up(sizeof(int2) * (size_t)(warps + 1), 256);
    s.bytes = s.off_bits + (n <= BITS_MAX_N ? align_up((size_t)(n + 31) / 32 * 4, 256) : 0);
    return s;
}

lrcc_status launch_gang(Ctx* c, const void* kernel, GangParams& P, int blocks, size_t smem) {
    if (smem) allow_smem(c, kernel, smem);
    GangCtl* gc = reinterpret_cast<GangCtl*>(reinterpret_cast<char*>(c->ctl) + offsetof(DevCtl, gang));
    DevCtl* ctl = c->ctl;
    void* args[] = {&P, &gc, &ctl};
    return cuda_status(cudaLaunchCooperativeKernel(kernel, dim3(blocks), dim3(GANG_THREADS), args, smem, c->stream));
}

}  // namespace

bool cc_gang_applies(const Plan& p) { return p.cc_hook == 1 && p.cc_max_rounds == 0 && p.use_graphs != 2; }

bool cc_one_block_applies(int64_t m, int64_t n) { return n <= ONE_MAX_N && m <= ONE_MAX_M; }

size_t cc_gang_ws(int64_t m, int64_t n, int sms, bool tight) {
    return cc_one_block_applies(m, n) ? 0 : gang_shape(m, n, sms, tight).bytes;
}

lrcc_status cc_run_gang(Ctx* c, const int32_t* src, const int32_t* dst, int64_t m, int64_t n, int32_t* label,
                        const Plan& p, bool tight) {
    if (cc_one_block_applies(m, n)) {
        const size_t smem = sizeof(int) * (size_t)n;
        allow_smem(c, (const void*)cc_one_block, sizeof(int) * ONE_MAX_N);
        phase_begin(c, c->stream);
        cc_one_block<<<1, GANG_THREADS, smem, c->stream>>>(src, dst, (int)m, (int)n, label, c->ctl);
        phase_end(c, c->stream, PH_CC_LOOP);
        return cuda_status(cudaGetLastError());
    }
    const GangShape S = gang_shape(m, n, c->sms, tight);
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
    // 14: 42 us without a sample, 57 with); from 16 edges per vertex and 2^22
    // vertices up half an edge per vertex is enough (R-MAT scale 24: 1.72 ms, 1.77
    // with one; scale 21: 314 us, 290 with one); with 1.5 edges per vertex half the
    // edges pay from 2^22 vertices on (2^24: 1111 against 1268 us; 2^20: 139
    // against 128).
    int64_t ms = m;
    if (p.cc_sample > 1) ms = m / p.cc_sample;
    else if (p.cc_sample < 0 && m >= (int64_t(1) << 19))
        ms = m >= 16 * n && n >= (int64_t(1) << 22) ? n / 2
             : m >= 2 * n ? n : n >= (int64_t(1) << 22) && 2 * m >= 3 * n ? m / 2 : m;
    P.ms = ms >= 4096 ? ms & ~int64_t(3) : m;
    P.first = P.ms;
    const bool sampled = P.ms < m;
    // Long passes over dense graphs: one pass that reads the parents forms the
    // giant (edges met later hook to what earlier ones made). In short ones most
    // edges are in flight at once, and three passes are needed (R-MAT scale 18: 83
    // us against 160), the first of which need not read the parents unless the
    // pass is long or the graph dense.
    P.sample_passes = m >= 8 * n && P.ms >= (int64_t(1) << 20) ? 1 : 3;
    P.first_min = sampled ? P.sample_passes > 1 && P.ms < (int64_t(1) << 22) : m <= 4 * n;
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
