// Batched connected components, hook rule 1: every graph by a gang of blocks
// (cc_gang.cuh) or, when it fits, by one block in shared memory.
//
// The large graphs used to be labelled together as one disjoint union by
// grid-wide passes: every pass streamed all edges and labels from HBM again, and
// most edges of every pass made two parent gathers and a hook. A gang finishes
// one graph before it takes the next, so a graph's parents stay in L2 from its
// first pass to its last, and its open edges are carried as pairs of roots. The
// table of the giant's members is left out: its 128 KB cost the other passes
// more in L1 than the filter gains (18.2 against 17.8 ms). 2048 uniform graphs of
// 2 edges per vertex, 2^8 to 2^20 vertices: 25.9 -> 17.1 ms (small graphs 0.95 ->
// 0.14). 64 of them of 2^17 vertices and more: 12.8 L2 requests per vertex at 181
// G/s, of the 290 that gathers alone reach (9.0 reads, 2.3 atomics and 1.3 writes); more
// blocks per SM or more gangs at once run the parents out of L2.
#include <algorithm>

#include "cc_gang.cuh"
#include "internal.h"

namespace lrcc {

namespace {

constexpr int SMALL_THREADS = 512;
constexpr int64_t SMALL_MAX_N = 16 << 10;   // one block's forest: 64 KB of shared memory
constexpr int64_t SMALL_MAX_M = 64 << 10;   // and the edges one block joins while others wait for it
constexpr size_t SMALL_SMEM = sizeof(int) * SMALL_MAX_N;
constexpr int GANG_MIN = 8;                 // blocks of a gang, at least
constexpr int CLASSES = 80;                 // small graphs by floor(log2(n + m)), then large ones

struct BatchPlan {
    int large;      // graphs for gangs: order[0 .. large)
    int gang;       // blocks per gang
};

// Sizes of graph k; whether its offsets are those of a graph.
__device__ __forceinline__ bool batch_graph(const int64_t* eoff, const int64_t* voff, int64_t k, int64_t total_edges,
                                            int64_t* n, int64_t* m) {
    *n = voff[k + 1] - voff[k];
    *m = eoff[k + 1] - eoff[k];
    return *n >= 0 && *n <= 0x7FFFFFFELL && *m >= 0 && *m <= 0x7FFFFFFFFFLL && voff[k] >= 0 && eoff[k] >= 0 &&
           eoff[k + 1] <= total_edges && (k > 0 || (voff[0] == 0 && eoff[0] == 0));
}

// Orders the graphs by size, largest first, those for gangs in front, and
// chooses the gang size: as many gangs as the largest graph leaves room for
// (the call lasts at least as long as that graph on its gang), of at least 8
// blocks. One block. A graph whose offsets are none (not from 0, decreasing, past
// total_edges) is reported and left out. scan_bad = 1 when vertex offsets decrease,
// so that graphs may overlap.
__global__ void __launch_bounds__(1024)
    cc_batch_order(const int64_t* __restrict__ eoff, const int64_t* __restrict__ voff, int64_t count,
                   int64_t total_edges, int blocks, int32_t* __restrict__ order, BatchPlan* plan, DevCtl* ctl) {
    __shared__ int s_hist[CLASSES], s_start[CLASSES];
    __shared__ unsigned long long s_total, s_most;
    for (int t = threadIdx.x; t < CLASSES; t += blockDim.x) s_hist[t] = 0;
    if (threadIdx.x == 0) s_total = s_most = 0;
    __syncthreads();
    auto klass = [&](int64_t k, unsigned long long* work) {
        int64_t n, m;
        *work = 0;
        if (!batch_graph(eoff, voff, k, total_edges, &n, &m)) {
            record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)k);
            if (n < 0) ctl->scan_bad = 1;
            return 0;
        }
        const int c = n + m <= 1 ? 0 : 63 - __clzll((unsigned long long)(n + m));
        if (n <= SMALL_MAX_N && m <= SMALL_MAX_M) return min(c, 39);
        *work = (unsigned long long)(n + m);
        return 40 + min(c, 39);
    };
    unsigned long long total = 0, most = 0, w;
    for (int64_t k = threadIdx.x; k < count; k += blockDim.x) {
        atomicAdd(&s_hist[klass(k, &w)], 1);
        total += w;
        most = max(most, w);
    }
    atomicAdd(&s_total, total);
    atomicMax(&s_most, most);
    __syncthreads();
    if (threadIdx.x == 0) {
        int run = 0;
        for (int c = CLASSES - 1; c >= 0; --c) {
            if (c == 39) plan->large = run;
            s_start[c] = run;
            run += s_hist[c];
        }
        const double share = s_total ? (double)s_most / (double)s_total * blocks : 0.0;
        int gang = min(blocks, GANG_MIN);
        while (gang < blocks && (double)gang < share) gang = min(blocks, gang + GANG_MIN);
        plan->gang = blocks / (blocks / gang);   // the blocks are shared out evenly
    }
    __syncthreads();
    for (int64_t k = threadIdx.x; k < count; k += blockDim.x)
        order[atomicAdd(&s_start[klass(k, &w)], 1)] = (int32_t)k;
}

// Whether graph k shares label entries with another graph (the whole block calls it).
__device__ bool overlaps(const int64_t* __restrict__ voff, int64_t count, int64_t k) {
    const int64_t b = voff[k], e = voff[k + 1];
    bool hit = false;
    for (int64_t i = threadIdx.x; i < count; i += blockDim.x) hit |= i != k && max(b, voff[i]) < min(e, voff[i + 1]);
    return __syncthreads_or(hit);
}

// One graph by the gang; false when a barrier gave up.
__device__ bool gang_label(const GangParams& P, Gang& G, DevCtl* ctl, volatile uint64_t* s_hook) {
    GangWork<false> w(P, G, ctl, s_hook, 0, 0);
    for (int64_t v = (int64_t)G.rank * GANG_THREADS + threadIdx.x; v < P.g.n; v += (int64_t)G.size * GANG_THREADS)
        P.g.p[v] = (int32_t)v;
    if (!G.sync()) return false;
    w.first_pass();
    if (!G.sync()) return false;
    w.template shortcut<false>(0);
    if (!G.sync()) return false;
    long long kept = w.settle(w.template star_pass<TABLE_NONE>(0, 0, nullptr));
    if (kept < 0) return false;
    if (P.ms < P.g.m) {
        for (int r = 2; r < P.sample_passes && kept > 0; ++r) {
            kept = w.settle(w.round());
            if (kept < 0) return false;
        }
        w.template shortcut<false>(0);
        if (!G.sync()) return false;
        const int left = w.act.count + (w.act.full ? 1 : 0);
        kept = w.settle(left + w.template star_pass<TABLE_NONE>(1, 0, nullptr));
        if (kept < 0) return false;
    }
    if (kept > 0 && !w.run_out(kept)) return false;
    if (w.lead()) atomicMax(&ctl->rounds, w.passes);
    return true;
}

__global__ void __launch_bounds__(GANG_THREADS, 1)
    cc_batch_gangs(const int32_t* __restrict__ src, const int32_t* __restrict__ dst, const int64_t* __restrict__ eoff,
                   const int64_t* __restrict__ voff, int64_t count, int64_t total_edges,
                   const int32_t* __restrict__ order, const BatchPlan* __restrict__ plan, GangCtl* gcs, int2* pairs,
                   int64_t pair_count, int32_t* label, DevCtl* ctl) {
    __shared__ int s_flag;
    __shared__ uint64_t s_hook[HOOK_SLOTS];
    __shared__ GangParams s_P;
    const int gang = plan->gang, gangs = (int)gridDim.x / gang, id = (int)blockIdx.x / gang;
    if (id >= gangs) return;
    GangCtl* gc = gcs + id;
    Gang G{gc, &gc->arrived[0], gang, (int)blockIdx.x % gang, 0, ctl, &s_flag};
    const int64_t room = pair_count / gangs;   // the gang's part of the pair buffer
    const int large = plan->large;
    for (;;) {
        if (G.rank == 0 && threadIdx.x == 0) {
            *(volatile unsigned*)&gc->instance = (unsigned)atomicAdd(&ctl->batch_next, 1);
            gc->kept[0] = gc->kept[1] = gc->kept[2] = 0;
        }
        if (!G.sync()) return;   // also: every block is done with the graph before
        const int q = (int)*(volatile unsigned*)&gc->instance;
        if (q >= large) return;
        // a graph's labels are its parents in local ids: gangs on graphs that share some
        // would follow each other's out of range
        if (ctl->scan_bad && overlaps(voff, count, order[q])) {
            if (!G.sync()) return;   // every block has read the instance
            continue;
        }
        if (threadIdx.x == 0) {
            const int64_t k = order[q];
            int64_t n, m;
            batch_graph(eoff, voff, k, total_edges, &n, &m);
            GangParams& P = s_P;
            P.g = GangGraph{src + eoff[k], dst + eoff[k], m, (int32_t)n, label + voff[k]};
            // A sample of 7/8 edge per vertex from 2 edges per vertex up. The first
            // pass reads the parents: its trees come out larger than those of linked
            // endpoints, which every later pass pays for here, where the gangs
            // together keep the L2 busy (17.8 ms against 18.6 for the 2048 graphs, both
            // with one sampled edge per vertex; with 7/8 17.4, with 5/4 1.2 ms more).
            P.ms = m >= 2 * n && m >= (int64_t(1) << 15) ? (n - n / 8) & ~int64_t(3) : m;
            P.first = P.ms;
            P.sample_passes = 3;
            P.first_min = false;
            P.buf = pairs + (int64_t)id * room;
            P.capw = (int)min(room / G.warps(), int64_t(1) << 30);
            P.bits = nullptr;
            P.left = nullptr;
            P.giant = nullptr;
            P.only = -1;
            int lg = 0;
            while ((int64_t(1) << lg) < n) ++lg;
            P.max_passes = 64 + 4 * lg;
            P.join = m < n ? min(int64_t(1) << 18, n / 8) : 0;
        }
        for (int h = threadIdx.x; h < HOOK_SLOTS; h += GANG_THREADS) s_hook[h] = ~0ull;
        __syncthreads();
        if (!gang_label(s_P, G, ctl, s_hook)) return;
    }
}

// The other graphs, one block each, largest first, in shared memory.
__global__ void __launch_bounds__(SMALL_THREADS)
    cc_batch_small(const int32_t* __restrict__ src, const int32_t* __restrict__ dst, const int64_t* __restrict__ eoff,
                   const int64_t* __restrict__ voff, int64_t count, int64_t total_edges,
                   const int32_t* __restrict__ order, const BatchPlan* __restrict__ plan, int32_t* __restrict__ label,
                   DevCtl* ctl) {
    extern __shared__ int small_p[];
    __shared__ int s_q;
    volatile int* p = small_p;
    const int first = plan->large;
    for (;;) {
        __syncthreads();   // the forest of the graph before is written out
        if (threadIdx.x == 0) s_q = atomicAdd(&ctl->seg_next, 1);
        __syncthreads();
        const int64_t q = (int64_t)first + s_q;
        if (q >= count) return;
        const int64_t k = order[q];
        int64_t n64, m64;
        if (!batch_graph(eoff, voff, k, total_edges, &n64, &m64) || n64 == 0) continue;
        const int n = (int)n64, m = (int)m64;
        const int32_t* s = src + eoff[k];
        const int32_t* d = dst + eoff[k];
        int32_t* out = label + voff[k];
        for (int v = threadIdx.x; v < n; v += SMALL_THREADS) p[v] = v;
        __syncthreads();
        for (int i = threadIdx.x; i < m; i += 4 * SMALL_THREADS) {
            int u[4], v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int e = i + j * SMALL_THREADS;
                u[j] = e < m ? __ldg(s + e) : 0;
                v[j] = e < m ? __ldg(d + e) : 0;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if ((uint32_t)u[j] >= (uint32_t)n || (uint32_t)v[j] >= (uint32_t)n)
                    record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)k);
                else
                    smem_join(p, u[j], v[j]);
            }
        }
        __syncthreads();
        for (int v = threadIdx.x; v < n; v += SMALL_THREADS) {
            int x = p[v];
            for (int y; (y = p[x]) != x;) x = y;
            out[v] = x;
        }
    }
}

// Pairs of all gangs: half the edges of the call (4 bytes per edge).
int64_t batch_pairs(int64_t total_edges) { return total_edges / 2; }

}  // namespace

bool cc_batch_gang_applies(const Plan& p) {
    return (p.cc_hook == 1 || p.cc_hook == 4) && p.cc_max_rounds == 0 && p.use_graphs != 2;
}

size_t cc_batch_gang_ws(int64_t count, int64_t total_edges, int sms) {
    return align_up(sizeof(int32_t) * (size_t)std::max<int64_t>(count, 1), 256) + 256 +
           align_up(sizeof(GangCtl) * (size_t)std::max(1, sms / GANG_MIN), 256) +
           align_up(sizeof(int2) * (size_t)batch_pairs(total_edges), 256);
}

lrcc_status cc_batch_gang_run(Ctx* c, const int32_t* src, const int32_t* dst, const int64_t* eoff, const int64_t* voff,
                              int64_t count, int64_t total_edges, int32_t* label) {
    cudaStream_t s = c->stream;
    char* w = static_cast<char*>(c->ws);
    int32_t* order = reinterpret_cast<int32_t*>(w);
    w += align_up(sizeof(int32_t) * (size_t)std::max<int64_t>(count, 1), 256);
    BatchPlan* plan = reinterpret_cast<BatchPlan*>(w);
    w += 256;
    GangCtl* gcs = reinterpret_cast<GangCtl*>(w);
    const size_t gcs_bytes = align_up(sizeof(GangCtl) * (size_t)std::max(1, c->sms / GANG_MIN), 256);
    w += gcs_bytes;
    int2* pairs = reinterpret_cast<int2*>(w);
    int64_t pair_count = batch_pairs(total_edges);
    const int blocks = c->sms;
    if (cudaMemsetAsync(gcs, 0, gcs_bytes, s) != cudaSuccess) return LRCC_ERR_CUDA;
    phase_begin(c, s);
    cc_batch_order<<<1, 1024, 0, s>>>(eoff, voff, count, total_edges, blocks, order, plan, c->ctl);
    phase_end(c, s, PH_BATCH_PREP);
    phase_begin(c, s);
    void* args[] = {&src, &dst, &eoff, &voff, &count, &total_edges, &order, &plan, &gcs, &pairs, &pair_count, &label, &c->ctl};
    const lrcc_status st = cuda_status(cudaLaunchCooperativeKernel((const void*)cc_batch_gangs, dim3(blocks),
                                                                   dim3(GANG_THREADS), args, 0, s));
    phase_end(c, s, PH_CC_LOOP);
    if (st != LRCC_OK) return st;
    phase_begin(c, s);
    allow_smem(c, (const void*)cc_batch_small, SMALL_SMEM);
    const int g = (int)std::min<int64_t>(count, persistent_grid(c, (const void*)cc_batch_small, SMALL_THREADS, SMALL_SMEM));
    cc_batch_small<<<g, SMALL_THREADS, SMALL_SMEM, s>>>(src, dst, eoff, voff, count, total_edges, order, plan, label, c->ctl);
    phase_end(c, s, PH_CC_BATCH);
    return cuda_status(cudaGetLastError());
}

}  // namespace lrcc
