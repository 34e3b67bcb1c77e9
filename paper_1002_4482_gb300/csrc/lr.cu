// List ranking kernels: Wyllie pointer jumping (Sec. 3.1, Algorithm 1) and the
// sparse ruling set / random splitter method (Sec. 3.2, Algorithms 2 and 3).
//
// Ruling set, as built here for sm_103a:
//   select   (RS1+RS2) one random splitter per block of D indices, at a hashed
//            offset, so a walk recognises it without a mark; the head is
//            splitter 0;
//   walk     (RS3) every splitter's sublist is walked once. Up to 2^24 elements
//            the walk reads succ and writes a 4-byte record (owner, position)
//            into the rank array (rs_walk_direct, rs_walk_lists), above it writes
//            what it visits as 32-byte chunks (rs_walk0c); weighted ranks walk
//            packed 8-byte words (rs_walk_values, rs_walk), split arrays are a
//            plan option (rs_walk0s);
//   recurse  (RS4) the list of splitters, weighted by sublist size, is again
//            cut by splitters and walked (rs_chase) until it fits one thread
//            block, which ranks it in shared memory (block_rank.cuh);
//   expand   (RS5) streaming passes turn (owner, position) into ranks.
// Every level stores the inclusive suffix weight S (elements from a node to
// the tail, itself included); the final rank is S - 1.
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <type_traits>

#include "block_rank.cuh"
#include "block_wyllie.cuh"
#include "common.cuh"
#include "gang.cuh"
#include "internal.h"
#include "list_block.cuh"

namespace lrcc {

namespace {

constexpr int BLOCK = 256;
constexpr int FINAL_THREADS = 1024;

// ------------------------------------------------------- shared-memory Wyllie

template <int PER>
__device__ __forceinline__ void cta_wyllie(int* val, int* nxt, int r, DevCtl* ctl) {
    block_wyllie<PER, FINAL_THREADS>(val, nxt, r, ctl);
}

// lr_rank_wyllie of a list of n <= PER * FINAL_THREADS elements: pointer
// jumping inside one block.
template <int PER>
__global__ void __launch_bounds__(FINAL_THREADS, 1)
    wy_small_kernel(const int32_t* __restrict__ succ, int n, int head, int32_t* __restrict__ rank, DevCtl* ctl) {
    extern __shared__ int sm[];
    int* val = sm;
    int* nxt = sm + PER * FINAL_THREADS;
    for (int i = threadIdx.x; i < n; i += FINAL_THREADS) {
        const int s = succ[i];
        const bool tail = (s == -1) | (s == i);
        const bool bad = !tail && (s < 0 || s >= n);
        if (bad) record_error(ctl, LRCC_ERR_INVALID_INPUT, i);
        nxt[i] = (tail || bad) ? (int)NIL : s;
        val[i] = 1;
    }
    __syncthreads();
    cta_wyllie<PER>(val, nxt, n, ctl);
    if (threadIdx.x == 0 && val[head] != n) record_error(ctl, LRCC_ERR_INVALID_INPUT, head);
    for (int i = threadIdx.x; i < n; i += FINAL_THREADS) rank[i] = val[i] - 1;
}

// Shared memory of a one-block ranking of r elements: the packed words and the
// splitters' two buffers.
constexpr size_t BR_SUB_BYTES = 2 * sizeof(uint2) * FINAL_THREADS;
constexpr size_t br_smem(int64_t r) { return sizeof(uint64_t) * (size_t)r + BR_SUB_BYTES; }

// One block ranks a whole list (block_rank.cuh). With weights (w != nullptr)
// it writes the inclusive suffix sums of w instead of the ranks.
__global__ void __launch_bounds__(FINAL_THREADS, 1)
    lr_small_kernel(const int32_t* __restrict__ succ, const int32_t* __restrict__ w, int n, int head,
                    int32_t* __restrict__ rank, uint32_t seed, DevCtl* ctl) {
    extern __shared__ __align__(16) unsigned char br_raw[];
    uint2* sub = reinterpret_cast<uint2*>(br_raw);
    uint64_t* W = reinterpret_cast<uint64_t*>(br_raw + BR_SUB_BYTES);
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += FINAL_THREADS) {
        const int s = succ[i];
        const bool tail = (s == -1) | (s == i);
        const bool bad = !tail && (s < 0 || s >= n);
        if (bad) record_error(ctl, LRCC_ERR_INVALID_INPUT, i);
        W[i] = pack((tail || bad) ? BR_NIL : (uint32_t)s, w ? (uint32_t)w[i] : 1u);
    }
    bool whole;
    const uint2* res = block_rank<FINAL_THREADS>(W, sub, n, head, seed, &whole, ctl);
    if (threadIdx.x == 0) {
        if (!whole) record_error(ctl, LRCC_ERR_INVALID_INPUT, head);
        clear_stats(ctl);   // a call of one launch has no memset before it
    }
    const int bias = w ? 0 : 1;
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += FINAL_THREADS) rank[i] = block_rank_sum<FINAL_THREADS>(W[i], res) - bias;
}

// Last ruling-set level: one block ranks the weighted list of splitters held
// in packed words R[j] = (next index or NIL, weight) and writes the inclusive
// suffix weights S. The head splitter (index 0) must see the whole list:
// `expect` elements, or, for weighted sums (expect < 0), whose total says
// nothing about the count, every one of the r splitters, whose walks must have
// reached `visited` elements (0: walks that mark what they visit).
__global__ void __launch_bounds__(FINAL_THREADS, 1)
    rs_final_kernel(const uint64_t* __restrict__ R, int r, int fixed, int32_t* __restrict__ S, int64_t expect,
                    unsigned long long visited, const int64_t* expect_dev, uint32_t seed, DevCtl* ctl) {
    if (ctl->scan_bad) return;
    if (expect_dev) expect = *expect_dev;
    if (fixed < r) r = min(r, fixed + ctl->ff_extra);   // extra owners in use (rs_walk_direct)
    extern __shared__ __align__(16) unsigned char br_raw[];
    uint2* sub = reinterpret_cast<uint2*>(br_raw);
    uint64_t* W = reinterpret_cast<uint64_t*>(br_raw + BR_SUB_BYTES);
#pragma unroll 4
    for (int j = threadIdx.x; j < r; j += FINAL_THREADS) {
        const uint64_t w = R[j];
        const uint32_t nx = lo32(w);
        if (nx >= (uint32_t)r && nx != NIL) record_error(ctl, LRCC_ERR_INVALID_INPUT, -3);
        W[j] = pack(nx < (uint32_t)r ? nx : BR_NIL, hi32(w));
    }
    bool whole;
    const uint2* res = block_rank<FINAL_THREADS>(W, sub, r, 0, seed, &whole, ctl);
    // with a total to expect, the head's total decides (it counts elements, and the
    // path from the head holds each once); splitters off the path are then empty ones
    if (threadIdx.x == 0 &&
        (expect >= 0 ? (int64_t)res[0].y != expect : !whole || (visited && ctl->visited != visited)))
        record_error(ctl, LRCC_ERR_INVALID_INPUT, -3);
#pragma unroll 4
    for (int j = threadIdx.x; j < r; j += FINAL_THREADS) S[j] = block_rank_sum<FINAL_THREADS>(W[j], res);
}

// ------------------------------------------------------------ ruling set

// Splitter choice (Sec. 3.2, RS2), stratified: the elements are cut into
// blocks of D = 2^logD consecutive indices and each block contributes exactly
// one splitter at a hashed offset, so a splitter's index is its block number
// and no compaction is needed. The head's block takes the head as its
// splitter, and block numbers are rotated so that the head is splitter 0.
// Offsets come from the MurmurHash3 finaliser of (block, seed).

// Level-0 select: one streaming pass packs succ into walk words
// W[i] = (next | SPL, splitter index) for splitters, (next, weight) for the
// rest (weight 1, or the element's value for weighted sums), and records each
// splitter's successor and weight. Warps stride over
// groups of 4 elements (Sec. 2.5), with 16-byte loads and stores.
template <bool VEC>
__global__ void __launch_bounds__(BLOCK)
    rs_select0(const int32_t* __restrict__ succ, const int32_t* __restrict__ val, int64_t n, int32_t head,
               uint64_t* __restrict__ W, int32_t* __restrict__ snext, int32_t* __restrict__ sw, int logD,
               int64_t nb, uint32_t seed, DevCtl* ctl, bool mark = true) {
    if (ctl->scan_bad) return;
    const uint64_t pol = policy_evict_first();
    const int64_t D = int64_t(1) << logD;
    const int64_t bh = head >> logD;
    const int64_t ngroups = (n + 3) >> 2;
    for (int64_t g = static_cast<int64_t>(blockIdx.x) * BLOCK + threadIdx.x; g < ngroups;
         g += static_cast<int64_t>(gridDim.x) * BLOCK) {
        const int64_t i0 = g * 4;
        int s[4], wt[4] = {1, 1, 1, 1};
        if (VEC && i0 + 3 < n) {
            const int4 v = ld_stream_v4(succ + i0, pol);
            s[0] = v.x; s[1] = v.y; s[2] = v.z; s[3] = v.w;
            if (val) {
                const int4 x = ld_stream_v4(val + i0, pol);
                wt[0] = x.x; wt[1] = x.y; wt[2] = x.z; wt[3] = x.w;
            }
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                s[q] = (i0 + q < n) ? ld_stream(succ + i0 + q, pol) : -1;
                if (val && i0 + q < n) wt[q] = ld_stream(val + i0 + q, pol);
            }
        }
        // D >= 4 and i0 % 4 == 0, so the 4 elements share one block
        const int64_t b = i0 >> logD;
        const uint32_t size = (uint32_t)min(D, n - (b << logD));
        const uint32_t off = b == bh ? (uint32_t)(head - (b << logD)) : block_offset((uint32_t)b, size, seed);
        const int64_t j = b >= bh ? b - bh : b - bh + nb;
        uint64_t w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t i = i0 + q;
            const int v = s[q];
            const bool tail = (v == -1) | (v == i);
            const bool bad = !tail && (v < 0 || v >= n);
            if (i < n && bad) record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)i);
            const uint32_t nx = (tail || bad) ? NIL : (uint32_t)v;
            if (mark && i < n && (uint32_t)(i - (b << logD)) == off) {
                w[q] = pack(nx | SPL, (uint32_t)j);
                snext[j] = (int32_t)nx;
                sw[j] = wt[q];
            } else {
                w[q] = pack(nx, (uint32_t)wt[q]);
            }
        }
        if (i0 + 3 < n) {
            ulonglong2* d = reinterpret_cast<ulonglong2*>(W + i0);
            d[0] = make_ulonglong2(w[0], w[1]);
            d[1] = make_ulonglong2(w[2], w[3]);
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i0 + q < n) W[i0 + q] = w[q];
        }
    }
}

// First-level splitters given by the caller (the even-splitter experiment of
// Sec. 3.2): spl[j] becomes splitter j of the words rs_select0 packed without
// splitters. spl[0] must be the head; an element out of range or given twice
// is reported (the first mark wins; the second finds SPL already set).
__global__ void __launch_bounds__(BLOCK)
    rs_mark_given(uint64_t* __restrict__ W, int64_t n, int32_t head, const int32_t* __restrict__ spl, int64_t r,
                  int32_t* __restrict__ snext, int32_t* __restrict__ sw, DevCtl* ctl) {
    for (int64_t j = static_cast<int64_t>(blockIdx.x) * BLOCK + threadIdx.x; j < r;
         j += static_cast<int64_t>(gridDim.x) * BLOCK) {
        const int32_t x = spl[j];
        if (x < 0 || x >= n || (j == 0 && x != head)) {
            record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)j);
            snext[j] = (int32_t)NIL;
            sw[j] = 0;
            continue;
        }
        unsigned int* lo = reinterpret_cast<unsigned int*>(W + x);   // low word of the element's packed word
        const unsigned int old = atomicOr(lo, SPL);
        if (old & SPL) {
            record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)j);
            snext[j] = (int32_t)NIL;
            sw[j] = 0;
            continue;
        }
        const unsigned int weight = reinterpret_cast<const unsigned int*>(W + x)[1];
        reinterpret_cast<unsigned int*>(W + x)[1] = (unsigned int)j;
        snext[j] = (int32_t)old;
        sw[j] = (int32_t)weight;
    }
}

// Brent's cycle detection for a walk that only reads: the anchor moves to the
// current element after 64, 128, 256, ... steps, so a walk caught in a cycle
// meets its anchor after at most three times the cycle's and its lead's length.
struct CycleGuard {
    uint32_t anchor, steps = 0, limit = 64;
    __device__ __forceinline__ explicit CycleGuard(uint32_t start) : anchor(start) {}
    // true when `cur` was visited before
    __device__ __forceinline__ bool seen(uint32_t cur) {
        if (cur == anchor) return true;
        if (++steps == limit) {
            anchor = cur;
            limit *= 2;
        }
        return false;
    }
};

// Sublist walk at level >= 1 (RS2 and RS3 in one kernel): the elements are the
// previous level's splitters with packed words R[i] = (next, weight), the head
// is element 0; elements from `fixed` on are extra owners of the first level,
// of which ctl->ff_extra are in use. Thread j starts at the splitter of block j, steps until the
// next element is a splitter (recognised by its hashed offset, so nothing has
// to be marked first), and stores P[i] = (prefix weight, owner) for every
// element it visits and Rout[j] = (next splitter, weight of its sublist).
//
// These levels are L2-resident and bound by the latency of the longest sublist
// (about D ln r steps), so a step is one dependent read of 304 cycles and
// little else: the splitter test of the next element runs while its word is on
// the way, one thread takes one sublist (no hand-out between steps), and the
// words read are not the words written. The form before marked the splitters
// in a pass of their own and overwrote R in place; a store to a line that was
// just read costs the L2 far more than a store elsewhere (read-then-store runs
// at 29-65 G/s, reads alone at 290, stores alone at 180-206).
//
// COUNT (weighted ranks, whose sums say nothing about how many elements they
// cover): the elements the walks reached are added up in *chased, which rs_expand
// compares with the level's size. That is enough: the level above is one list
// holding all its elements (its own count, or the last level's), so the walks of
// this one end at different splitters, cannot meet, and reach each element at
// most once.
static_assert(sizeof(DevCtl::chased) >= MAX_LEVELS * sizeof(unsigned long long), "a count for every level");
template <bool COUNT>
__global__ void __launch_bounds__(BLOCK)
    rs_chase(const uint64_t* __restrict__ R, uint32_t nl, uint64_t* __restrict__ P, uint64_t* __restrict__ Rout,
             uint32_t r, int logD, uint32_t seed, uint32_t fixed, unsigned long long* chased, DevCtl* ctl) {
    if (ctl->scan_bad) return;
    const uint32_t j = blockIdx.x * BLOCK + threadIdx.x;
    const uint32_t D = 1u << logD;
    auto offset = [&](uint32_t b) {
        return b == 0 ? 0u : block_offset(b, min(D, nl - (b << logD)), seed);
    };
    // walks sublist j; the elements it reached
    auto walk = [&]() -> uint32_t {
        const uint32_t start = (j << logD) + offset(j);
        if (start >= fixed && start - fixed >= (uint32_t)ctl->ff_extra) {   // an extra owner nobody took
            Rout[j] = pack(NIL, 0);
            return 0;
        }
        uint64_t w = R[start];
        P[start] = pack(0, j);
        uint32_t cur = lo32(w), pre = hi32(w), steps = 1;
        CycleGuard guard(start);
        uint32_t next = NIL;
        while (cur != NIL) {
            if (cur >= nl || guard.seen(cur)) {
                record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)cur);
                break;
            }
            w = R[cur];
            const uint32_t b = cur >> logD;
            if ((cur & (D - 1)) == offset(b)) {
                next = b;
                break;
            }
            P[cur] = pack(pre, j);
            pre += hi32(w);
            if (COUNT) ++steps;
            cur = lo32(w);
        }
        Rout[j] = pack(next, pre);
        return steps;
    };
    if (!COUNT) {
        if (j < r) walk();
        return;
    }
    unsigned long long reached = j < r ? walk() : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) reached += __shfl_xor_sync(0xffffffffu, reached, o);
    if ((threadIdx.x & 31) == 0 && reached) atomicAdd(chased, reached);
}

// Sublist walk (RS3). Each thread keeps K walks in flight so that K
// independent gathers are outstanding; a warp claims splitters in chunks of
// 64 with one atomic and hands them to lanes as their walks end, which
// balances the geometric spread of sublist lengths.
template <int K>
__global__ void __launch_bounds__(BLOCK)
    rs_walk(uint64_t* __restrict__ W, const int32_t* __restrict__ snext, const int32_t* __restrict__ sw,
            uint64_t* __restrict__ Rout, int r, int* work, int64_t nlevel, DevCtl* ctl) {
    if (ctl->scan_bad) return;
    constexpr int CHUNK = 64;
    const int lane = threadIdx.x & 31;
    int pool = 0, pool_end = 0;
    bool exhausted = false;
    int j[K];
    uint32_t cur[K], pre[K];
    int64_t steps[K];
#pragma unroll
    for (int q = 0; q < K; ++q) {
        j[q] = -1;
        cur[q] = NIL;
        pre[q] = 0;
        steps[q] = 0;
    }
    for (;;) {
#pragma unroll
        for (int q = 0; q < K; ++q) {
            bool need = j[q] < 0;
            unsigned m = __ballot_sync(0xffffffffu, need);
            while (m && !exhausted) {
                if (pool >= pool_end) {
                    int b = 0;
                    if (lane == 0) b = atomicAdd(work, CHUNK);
                    b = __shfl_sync(0xffffffffu, b, 0);
                    if (b >= r) {
                        exhausted = true;
                        break;
                    }
                    pool = b;
                    pool_end = min(b + CHUNK, r);
                }
                const int avail = pool_end - pool;
                const int rk = __popc(m & lanemask_lt());
                if (need && rk < avail) {
                    const int jj = pool + rk;
                    j[q] = jj;
                    cur[q] = (uint32_t)snext[jj];
                    pre[q] = (uint32_t)sw[jj];
                    steps[q] = 0;
                    need = false;
                }
                pool += min(avail, __popc(m));
                m = __ballot_sync(0xffffffffu, need);
            }
        }
        bool act = false;
#pragma unroll
        for (int q = 0; q < K; ++q) act |= j[q] >= 0;
        if (!__any_sync(0xffffffffu, act)) break;
        uint64_t w[K];
#pragma unroll
        for (int q = 0; q < K; ++q)
            w[q] = (j[q] >= 0 && cur[q] < (uint32_t)nlevel) ? W[cur[q]] : 0ull;
#pragma unroll
        for (int q = 0; q < K; ++q) {
            if (j[q] < 0) continue;
            if (cur[q] == NIL) {
                Rout[j[q]] = pack(NIL, pre[q]);
                j[q] = -1;
                continue;
            }
            const uint32_t lo = lo32(w[q]), hi = hi32(w[q]);
            if (cur[q] >= (uint32_t)nlevel || (!(lo & SPL) && ((hi & VIS) || ++steps[q] > nlevel))) {
                record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)cur[q]);
                Rout[j[q]] = pack(NIL, pre[q]);
                j[q] = -1;
            } else if (lo & SPL) {
                Rout[j[q]] = pack(hi, pre[q]);
                j[q] = -1;
            } else {
                W[cur[q]] = pack(pre[q], (uint32_t)j[q] | VIS);
                pre[q] += hi;
                cur[q] = lo;
            }
        }
    }
}

// Ceiling of the first-level walk's access pattern: dependent 4-byte reads of
// succ, with the walk's load form and none of its bookkeeping (no chunk
// writes, no splitter test). Chain c of `chains` starts at element
// floor(c * n / chains) and takes `steps` steps; a chain that reaches a tail
// (or an id outside [0, n)) continues from a hashed element, which costs no
// read. Each thread advances PROBE_K chains together, as the walk does; the
// wrapped sum of the elements reached goes to *out, so no load is dropped.
constexpr int PROBE_K = 4;
__global__ void __launch_bounds__(BLOCK)
    rs_chase_probe(const int32_t* __restrict__ succ, int64_t n, int64_t chains, int64_t steps,
                   unsigned long long* out) {
    const int64_t c0 = ((int64_t)blockIdx.x * BLOCK + threadIdx.x) * PROBE_K;
    int64_t cur[PROBE_K];
    bool live[PROBE_K];
#pragma unroll
    for (int q = 0; q < PROBE_K; ++q) {
        live[q] = c0 + q < chains;
        cur[q] = live[q] ? (c0 + q) * n / chains : 0;   // c < 2^31 and n <= 2^31: no overflow
    }
    unsigned long long acc = 0;
    for (int64_t k = 0; k < steps; ++k) {
        int32_t nx[PROBE_K];
#pragma unroll
        for (int q = 0; q < PROBE_K; ++q) nx[q] = live[q] ? __ldg(succ + cur[q]) : 0;
#pragma unroll
        for (int q = 0; q < PROBE_K; ++q) {
            if (!live[q]) continue;
            int64_t x = nx[q];
            if (x < 0 || x >= n || x == cur[q])
                x = (int64_t)(((uint64_t)mix32((uint32_t)cur[q] ^ (uint32_t)k * 0x9E3779B9u) * (uint64_t)n) >> 32);
            acc += (unsigned long long)x;
            cur[q] = x;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(out, acc);
}

// ------------------------------------------------ level 0, read-only walk
//
// Random HBM accesses are limited by row activations, not bytes: a random
// read costs one activation, a random read-modify-write two. This level-0
// path therefore walks succ READ-ONLY (one activation per element) and never
// writes a per-element word at a random place:
//   walk     each walk buffers the elements it visits in registers and
//            writes them 8 at a time as one 32-byte chunk (ids in visiting
//            order, plus (first position k0, owner j)) into its block's
//            region; the block also counts its elements per coarse id
//            bucket (NBK buckets of consecutive ids);
//   scan     the per-(bucket, block) counts become output offsets;
//   scatter  each block turns its chunks into (element, rank) pairs with one
//            gather of the owner's suffix weight per chunk, written grouped
//            by bucket;
//   place    the pairs, in bucket order, write rank[element]; the writes of
//            one bucket fall in a window of a few MB that stays in L2, so
//            lines are complete before they are written back.
// A walk that runs longer than `careful` steps marks the elements it visits
// in a bitmap and stops with an error on a repeat, so a cycle without a
// splitter cannot trap it; valid lists never repeat an element.

constexpr int CIDS = 8;        // element ids per chunk (one 32-byte sector)
// Coarse id buckets of the scatter (a bucket's rank writes stay in L2 while
// rs_place works through it). More buckets make each round's runs shorter:
// with 1024 buckets at 2^28 elements the scatter took 2.67 ms instead of 1.41.
constexpr int NBK_LOG = 8;
constexpr int NBK = 1 << NBK_LOG;
constexpr int NSEG = 4;        // scatter work units per walk block region

struct Level0 {
    int64_t n, nb, bh;   // elements, splitters (blocks), the head's block
    int logD;
    uint32_t head_off;   // offset of the head inside its block
    uint32_t seed;
    // batched lists ranked as one list (see lr_enqueue_rs): the first list's
    // head, read on the device (bh and head_off are derived from it), and the
    // heads of the other lists that are extra splitters nb, nb + 1, ...
    const int64_t* head_dev = nullptr;
    const int32_t* extra = nullptr;
    const int* extra_count = nullptr;
};

struct Chunks {
    int32_t* ids;        // chunk c: ids[8c .. 8c+8), unused slots -1
    uint64_t* meta;      // meta[c] = k0 << 32 | j
    int* fill;           // chunks written into each block's own region
    int* counts;         // [NBK][units] elements per (bucket, scatter unit); then row offsets
    int* totals;         // [NBK] elements per bucket
    uint32_t* vis;       // careful-mode marks, one bit per element
    int64_t cap;         // chunks per block region (NSEG segments of segcap)
    int segcap;          // chunks per segment (even); a segment is one scatter work unit
    int units;           // scatter units: NSEG per block region, then the overflow pool's segments
    int64_t ovf_cap;     // overflow chunks
    int64_t ovf_base;    // index of the first overflow chunk (= grid * cap)
    int shift;           // coarse bucket of element x = x >> shift
    int64_t careful;     // steps after which a walk marks what it visits
};

// Index of x among the level-0 splitters, or -1 if x is not one.
__device__ __forceinline__ int64_t splitter_index0(int64_t x, const Level0& L0) {
    const int64_t D = int64_t(1) << L0.logD;
    const int64_t b = x >> L0.logD;
    const uint32_t size = (uint32_t)min(D, L0.n - (b << L0.logD));
    const uint32_t off = b == L0.bh ? L0.head_off : block_offset((uint32_t)b, size, L0.seed);
    if ((uint32_t)(x - (b << L0.logD)) != off) return -1;
    return b >= L0.bh ? b - L0.bh : b - L0.bh + L0.nb;
}

// Element of splitter j.
__device__ __forceinline__ int64_t splitter_node0(int64_t j, const Level0& L0) {
    if (j >= L0.nb) return L0.extra[j - L0.nb];
    const int64_t D = int64_t(1) << L0.logD;
    int64_t b = j + L0.bh;
    if (b >= L0.nb) b -= L0.nb;
    const uint32_t size = (uint32_t)min(D, L0.n - (b << L0.logD));
    const uint32_t off = b == L0.bh ? L0.head_off : block_offset((uint32_t)b, size, L0.seed);
    return (b << L0.logD) + off;
}

// 32-bit level-0 geometry (element ids are int32, so n < 2^31).
struct Geo32 {
    uint32_t n, nb, bh, head_off, seed, D;
    int logD;
};
__device__ __forceinline__ Geo32 geo32(const Level0& L0) {
    Geo32 g;
    g.n = (uint32_t)L0.n;
    g.nb = (uint32_t)L0.nb;
    g.bh = (uint32_t)L0.bh;
    g.head_off = L0.head_off;
    g.seed = L0.seed;
    g.logD = L0.logD;
    g.D = 1u << L0.logD;
    return g;
}
// offset of the splitter inside block b (the same value block_offset gives)
__device__ __forceinline__ uint32_t block_off32(uint32_t b, const Geo32& g) {
    if (b == g.bh) return g.head_off;
    const uint32_t base = b << g.logD;
    const uint32_t size = min(g.D, g.n - base);
    return __umulhi(mix32(b * 0x9E3779B1u + g.seed), size);
}
// index of x among the level-0 splitters, or -1
__device__ __forceinline__ int splitter_index32(uint32_t x, const Geo32& g) {
    const uint32_t b = x >> g.logD;
    if ((x & (g.D - 1)) != block_off32(b, g)) return -1;
    return (int)(b >= g.bh ? b - g.bh : b - g.bh + g.nb);
}
__device__ __forceinline__ uint32_t splitter_node32(uint32_t j, const Geo32& g, const int32_t* extra) {
    if (j >= g.nb) return (uint32_t)extra[j - g.nb];
    uint32_t b = j + g.bh;
    if (b >= g.nb) b -= g.nb;
    return (b << g.logD) + block_off32(b, g);
}

// Read-only sublist walk (RS3). Warps claim splitters in chunks of 64 and
// hand them to lanes as their walks end (the hardware scheduler then
// balances the uneven sublists, Sec. 3.2). Element arithmetic is 32-bit (ids
// are int32) and the ids a walk collects for its next chunk wait in shared
// memory: against 64-bit indices and an 8-entry register buffer, 7 % faster at
// 2^25 elements, 0.6 % at 2^28, where the random reads of succ bound it.
template <int K>
__global__ void __launch_bounds__(BLOCK)
    rs_walk0c(const int32_t* __restrict__ succ, Level0 L0, Chunks C, uint64_t* __restrict__ R1, int* work,
              DevCtl* ctl) {
    if (L0.head_dev) {
        if (!L0.head_dev[3]) return;   // batched lists that this form does not rank
        const int64_t gh = *L0.head_dev;
        L0.bh = gh >> L0.logD;
        L0.head_off = (uint32_t)(gh - (L0.bh << L0.logD));
    }
    const Geo32 g = geo32(L0);
    constexpr int WCHUNK = 64;   // splitters a warp claims at once (32 and 128: no faster)
    __shared__ int s_fill;
    __shared__ int s_cnt[NSEG][NBK];
    // the ids a walk has visited since its last flush: slot t of chain q of thread i at
    // s_ids[(q * CIDS + t) * BLOCK + i] (one bank per thread)
    __shared__ int32_t s_ids[K * CIDS * BLOCK];
    for (int t = threadIdx.x; t < NSEG * NBK; t += BLOCK) (&s_cnt[0][0])[t] = 0;
    if (threadIdx.x == 0) s_fill = 0;
    __syncthreads();
    const uint32_t r = g.nb + (L0.extra_count ? (uint32_t)*L0.extra_count : 0u);
    const int lane = threadIdx.x & 31;
    int pool = 0, pool_end = 0;
    bool exhausted = false;
    int j[K];
    uint32_t cur[K], k[K], k0[K];
    int bn[K];
#pragma unroll
    for (int q = 0; q < K; ++q) {
        j[q] = -1;
        cur[q] = 0;
        k[q] = k0[q] = 0;
        bn[q] = 0;
    }
    for (;;) {
#pragma unroll
        for (int q = 0; q < K; ++q) {
            bool need = j[q] < 0;
            unsigned m = __ballot_sync(0xffffffffu, need);
            while (m && !exhausted) {
                if (pool >= pool_end) {
                    int b = 0;
                    if (lane == 0) b = atomicAdd(work, WCHUNK);
                    b = __shfl_sync(0xffffffffu, b, 0);
                    if ((uint32_t)b >= r) {
                        exhausted = true;
                        break;
                    }
                    pool = b;
                    pool_end = (int)min((uint32_t)b + WCHUNK, r);
                }
                const int avail = pool_end - pool;
                const int rk = __popc(m & lanemask_lt());
                if (need && rk < avail) {
                    j[q] = pool + rk;
                    cur[q] = splitter_node32((uint32_t)j[q], g, L0.extra);
                    k[q] = k0[q] = 0;
                    bn[q] = 0;
                    need = false;
                }
                pool += min(avail, __popc(m));
                m = __ballot_sync(0xffffffffu, need);
            }
        }
        bool act = false;
#pragma unroll
        for (int q = 0; q < K; ++q) act |= j[q] >= 0;
        if (!__any_sync(0xffffffffu, act)) break;
        int32_t nx[K];
        // read-only loads at normal L2 priority: the part of succ that L2 holds (an
        // eighth at 2^28) then serves repeat visits; evict-first loads gave those
        // hits up and made the walk 5 % slower
#pragma unroll
        for (int q = 0; q < K; ++q) nx[q] = j[q] >= 0 ? __ldg(succ + cur[q]) : -1;
#pragma unroll
        for (int q = 0; q < K; ++q) {
            if (j[q] < 0) continue;
            bool end = false, bad = false;
            if (k[q] >= C.careful) {
                const uint32_t bit = 1u << (cur[q] & 31);
                if (atomicOr(C.vis + (cur[q] >> 5), bit) & bit) bad = true;   // element reached twice
            }
            s_ids[(q * CIDS + bn[q]) * BLOCK + threadIdx.x] = (int32_t)cur[q];
            ++bn[q];
            const int32_t x = nx[q];
            uint64_t rw = 0;
            if (bad) {
                end = true;
            } else if (x == -1 || (uint32_t)x == cur[q]) {
                rw = pack(NIL, k[q] + 1);
                end = true;
            } else if (x < 0 || (uint32_t)x >= g.n) {
                bad = end = true;
            } else {
                const int sj = splitter_index32((uint32_t)x, g);
                if (sj >= 0) {
                    rw = pack((uint32_t)sj, k[q] + 1);
                    end = true;
                }
            }
            if (bad) {
                record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)cur[q]);
                rw = pack(NIL, k[q] + 1);
            }
            if (bn[q] == CIDS || end) {
                // flush one chunk: own region first, then the shared overflow pool
                const int slot = atomicAdd(&s_fill, 1);
                int64_t c = -1;
                int ovf_unit = -1;   // scatter unit of an overflow chunk (counted in global memory)
                if (slot < C.cap) {
                    c = (int64_t)blockIdx.x * C.cap + slot;
                } else {
                    const int o = atomicAdd(&ctl->ovf_next, 1);
                    if (o < C.ovf_cap) {
                        c = C.ovf_base + o;
                        ovf_unit = (int)gridDim.x * NSEG + o / C.segcap;
                    } else {
                        record_error(ctl, LRCC_ERR_INVALID_INPUT, -4);
                    }
                }
                if (c >= 0) {
                    const int seg = slot / C.segcap;
                    int32_t v[CIDS];
#pragma unroll
                    for (int t = 0; t < CIDS; ++t)
                        v[t] = t < bn[q] ? s_ids[(q * CIDS + t) * BLOCK + threadIdx.x] : -1;
                    // streaming stores: the chunks are read once, by the scatter, and
                    // should not push succ out of L2; one 32-byte store per chunk (chunks
                    // are 32-byte aligned) moves a whole sector in one request instead of
                    // two 16-byte halves (5.55 -> 5.51 ms at 2^28)
                    st_cs_v8(C.ids + c * CIDS, v);
                    __stcs(reinterpret_cast<unsigned long long*>(C.meta + c),
                           (unsigned long long)((static_cast<uint64_t>(k0[q]) << 32) | static_cast<uint32_t>(j[q])));
#pragma unroll
                    for (int t = 0; t < CIDS; ++t)
                        if (t < bn[q]) {
                            if (ovf_unit < 0) atomicAdd(&s_cnt[seg][v[t] >> C.shift], 1);
                            else atomicAdd(&C.counts[(int64_t)(v[t] >> C.shift) * C.units + ovf_unit], 1);
                        }
                }
                k0[q] = k[q] + 1;
                bn[q] = 0;
            }
            if (end) {
                R1[j[q]] = rw;
                j[q] = -1;
            } else {
                cur[q] = (uint32_t)x;
                ++k[q];
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) C.fill[blockIdx.x] = min(s_fill, (int)C.cap);
    for (int t = threadIdx.x; t < NSEG * NBK; t += BLOCK) {
        const int bk = t % NBK, seg = t / NBK;
        C.counts[(int64_t)bk * C.units + (int64_t)blockIdx.x * NSEG + seg] = s_cnt[seg][bk];
    }
}

// Exclusive scan of each bucket's row of per-block counts, in place, one
// block per bucket; the row total goes to totals[bucket]. The start of each
// bucket (a scan over NBK totals) is formed by the scatter blocks themselves.
constexpr int SCAN_THREADS = 256;
__device__ __forceinline__ void scan_counts(int* counts, int G, int* totals) {
    __shared__ int s_warp[SCAN_THREADS / 32];
    int* row = counts + (int64_t)blockIdx.x * G;
    const int per = (G + SCAN_THREADS - 1) / SCAN_THREADS;
    const int b = threadIdx.x * per, e = min(G, b + per);
    int sum = 0;
    for (int i = b; i < e; ++i) sum += row[i];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) s_warp[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        int v = lane < SCAN_THREADS / 32 ? s_warp[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += t;
        }
        if (lane < SCAN_THREADS / 32) s_warp[lane] = v;
    }
    __syncthreads();
    int run = (wid ? s_warp[wid - 1] : 0) + incl - sum;
    for (int i = b; i < e; ++i) {
        const int c = row[i];
        row[i] = run;
        run += c;
    }
    if (threadIdx.x == SCAN_THREADS - 1) totals[blockIdx.x] = run;
}
__global__ void __launch_bounds__(SCAN_THREADS) rs_scan_counts(int* counts, int G, int* totals) {
    scan_counts(counts, G, totals);
}

// Chunks of walk block g -> (element, rank) pairs at block g's offsets of
// each bucket. Radix-partition style, in rounds of SC_CHUNKS chunks: the
// round's chunk ids and headers arrive in shared memory by bulk copy, the
// round's elements are ranked by bucket with shared atomics, their
// (element, rank) pairs laid out sorted by bucket in a tile, and every
// bucket's run is written with coalesced stores at the block's next offset
// for that bucket. The phases of a round are separated by block barriers and
// the kernel is bound by their latency, not by shared-memory bandwidth, so
// blocks per SM count most: at 2^28 elements a 16-bit slot-index tile with 4
// blocks per SM took 1.44 ms, the pair tile with two staging buffers (2 blocks
// per SM) 1.38 ms, rounds of 3 chunks per thread 1.47 ms, and the pair tile
// with one staging buffer (3 blocks per SM) 1.22 ms. Blocks
// are persistent and take work units u = blockIdx.x, + gridDim.x, ...: the
// NSEG segments of every walk block's region, then the segments of the shared
// overflow pool (each unit's per-bucket counts come from the walk).
// Compile-time shape of a round: chunks per thread (SC_U), staging buffers
// (SC_BUF) and the blocks per SM the launch bounds ask for. Rounds of one chunk
// per thread with two or three buffers and 4-6 blocks per SM took 1.54-1.78 ms
// at 2^28 against 1.21 ms for the default: a round's fixed cost (barriers, the
// scan, the owners' gathers) is paid per round, so fewer, larger rounds win.
#ifndef LRCC_SC_U
#define LRCC_SC_U 2
#endif
#ifndef LRCC_SC_BUF
#define LRCC_SC_BUF 1
#endif
#ifndef LRCC_SC_MINB
#define LRCC_SC_MINB 3
#endif

constexpr int SC_U = LRCC_SC_U;                 // chunks per thread and round
// One staging buffer: a round's ids and headers move into registers in its
// first phase, and the next round's bulk copy lands in the same buffer while
// this round is scanned and written out (0.35 against 0.40 ms at 2^26). With
// more buffers, the copy issued after round k's first phase is round k + SC_BUF.
constexpr int SC_BUF = LRCC_SC_BUF;
constexpr int SC_CHUNKS = SC_U * BLOCK;         // chunks per round
constexpr int SC_ITEMS = SC_CHUNKS * CIDS;      // element slots per round
// Polls of a bulk-copy barrier before giving up. A poll that finds the phase
// open suspends the thread for a few microseconds (about 4.3 us measured on
// GB300), so the limit is about one second.
constexpr int SC_WAIT_LIMIT = 1 << 18;
struct ScatterSmem {
    int32_t ids[SC_BUF][SC_ITEMS];      // chunk ids of the round in each buffer
    uint64_t meta[SC_BUF][SC_CHUNKS];   // chunk headers (k0 << 32 | owner)
    uint64_t tile[SC_ITEMS];       // the round's (element, rank) pairs sorted by bucket
    int cnt[NBK];                  // elements per bucket in the round
    int delta[NBK];                // pair position minus tile slot, per bucket, in the round
    int tstart[NBK];               // start of each bucket's run in the tile
    int warp[BLOCK / 32];
    uint64_t bar[SC_BUF];
};
constexpr size_t SC_SMEM = sizeof(ScatterSmem);

// The 8 ids of one chunk from shared memory. Lanes 4-7 of every 8 read the
// two 16-byte halves in the other order, so that each quarter-warp phase of
// the 16-byte loads touches all 32 banks once.
__device__ __forceinline__ void load_chunk(const int32_t* p, int32_t (&id)[CIDS]) {
    const int sw = (threadIdx.x >> 2) & 1;
    const int4* src = reinterpret_cast<const int4*>(p);
    const int4 a = src[sw], d = src[sw ^ 1];
    const int4 lo = sw ? d : a, hi = sw ? a : d;
    id[0] = lo.x; id[1] = lo.y; id[2] = lo.z; id[3] = lo.w;
    id[4] = hi.x; id[5] = hi.y; id[6] = hi.z; id[7] = hi.w;
}

__global__ void __launch_bounds__(BLOCK, LRCC_SC_MINB)
    rs_scatter(Chunks C, int G, const int32_t* __restrict__ S1, uint64_t* __restrict__ pairs, int64_t n,
               DevCtl* ctl) {
    extern __shared__ __align__(128) unsigned char sc_raw[];
    ScatterSmem& s = *reinterpret_cast<ScatterSmem*>(sc_raw);
    static_assert(NBK == BLOCK, "one thread per bucket");
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    // block-wide exclusive scan of one value per thread (uses s.warp; one sync).
    // Every caller passes another block barrier before the next scan rewrites
    // s.warp, so the scan needs no barrier after reading it.
    auto block_scan = [&](int v, int* total) {
        int incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        if (lane == 31) s.warp[wid] = incl;
        __syncthreads();
        int off = 0, all = 0;
#pragma unroll
        for (int w = 0; w < BLOCK / 32; ++w) {
            const int x = s.warp[w];
            off += w < wid ? x : 0;
            all += x;
        }
        *total = all;
        return off + incl - v;
    };
    int bstart;                     // start of bucket t in the pair array
    {
        int all = 0;
        bstart = block_scan(C.totals[t], &all);
        if (all == 0) return;   // nothing was walked (and ctl->pairs is 0)
        if (blockIdx.x == 0 && t == 0) ctl->pairs = all;
    }
    s.cnt[t] = 0;
    if (t == 0) {
        for (int b = 0; b < SC_BUF; ++b) mbar_init(&s.bar[b], 1);
        fence_proxy_async_smem();   // the initialised barriers are visible to the bulk copies
    }
    __syncthreads();
    // L2 hints: the chunks are read and the pairs written once (evict first),
    // while the owners' suffix ranks S1 (4 bytes per splitter) are gathered
    // once per chunk and should stay (evict last): 1.17 against 1.20 ms at 2^28
    const uint64_t pol = policy_evict_first();
    const uint64_t keep = policy_evict_last();
    uint32_t phase = 0;             // bit b: parity of the next completion of buffer b's barrier
    uint32_t in_flight = 0;         // bit b: a copy into buffer b is not yet waited for (thread 0)
    bool failed = false;
    int my_base = 0;                // next free pair of bucket t (this thread's) in the current unit

    // issue the bulk copy of round k of region g (chunks own0 + k*SC_CHUNKS ..) into buffer b
    auto issue = [&](int64_t first, int nf, int k, int b) {
        const int64_t c0 = first + (int64_t)k * SC_CHUNKS;
        const int cnt = min(SC_CHUNKS, nf - k * SC_CHUNKS);
        const int cm = (cnt + 1) & ~1;   // headers in pairs: 16-byte multiple (segments are even)
        const uint32_t bi = (uint32_t)cnt * CIDS * 4u, bm = (uint32_t)cm * 8u;
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(&s.bar[b], bi + bm);
        bulk_g2s(s.ids[b], C.ids + c0 * CIDS, bi, &s.bar[b], pol);
        bulk_g2s(s.meta[b], C.meta + c0, bm, &s.bar[b], pol);
        in_flight |= 1u << b;
    };

    // one round over buffer b, whose chunks [0, cnt) are valid (a chunk whose
    // first id is -1 is empty)
    auto process = [&](int b, int cnt, int64_t uc0, int unf, int knext) {
        // the owners' suffix ranks (L2 gathers) are issued first, so their latency
        // overlaps the counting and the scan
        int32_t top[SC_U];
#pragma unroll
        for (int u = 0; u < SC_U; ++u) {
            const int c = u * BLOCK + t;
            const uint64_t mt = s.meta[b][c];
            top[u] = (c < cnt && s.ids[b][c * CIDS] >= 0) ? ld_nc_hint(S1 + lo32(mt), keep) - 1 - (int32_t)hi32(mt) : 0;
        }
        int32_t id[SC_U][CIDS];
        int loc[SC_U][CIDS];
#pragma unroll
        for (int u = 0; u < SC_U; ++u) {
            const int c = u * BLOCK + t;
            load_chunk(&s.ids[b][c * CIDS], id[u]);
#pragma unroll
            for (int q = 0; q < CIDS; ++q) {
                if (c >= cnt) id[u][q] = -1;
                loc[u][q] = id[u][q] >= 0 ? atomicAdd(&s.cnt[id[u][q] >> C.shift], 1) : 0;
            }
        }
        fence_proxy_async_smem();   // this thread's reads of the buffer come before the next copy into it
        __syncthreads();
        // the round's ids and headers now sit in registers: the copy of round
        // k + SC_BUF goes into this buffer while this round is scanned and written out
        if (t == 0 && knext >= 0) issue(uc0, unf, knext, b);
        const int h = s.cnt[t];
        s.cnt[t] = 0;               // counts of the next round
        int items = 0;
        const int ts = block_scan(h, &items);
        s.tstart[t] = ts;
        s.delta[t] = my_base - ts;     // pair position of tile slot i of bucket t: delta[t] + i
        my_base += h;
        __syncthreads();
#pragma unroll
        for (int u = 0; u < SC_U; ++u)
#pragma unroll
            for (int q = 0; q < CIDS; ++q)
                if (id[u][q] >= 0)
                    s.tile[s.tstart[id[u][q] >> C.shift] + loc[u][q]] =
                        pack((uint32_t)id[u][q], (uint32_t)(top[u] - q));
        __syncthreads();
        for (int i = t; i < items; i += BLOCK) {
            const uint64_t pr = s.tile[i];
            const int64_t pos = (int64_t)s.delta[lo32(pr) >> C.shift] + i;
            if (pos < n) st_hint_u64(pairs + pos, pr, pol);
        }
        // no barrier here: the next round rebuilds the tile only after its own
        // barriers (the bounded wait's __syncthreads_or comes first, and a new
        // unit starts with one)
    };

    const int64_t no_all = min((int64_t)ctl->ovf_next, C.ovf_cap);
    const int own_units = G * NSEG;
    for (int unit = blockIdx.x; unit < C.units && !failed; unit += gridDim.x) {
        int nf;
        int64_t c0;
        if (unit < own_units) {
            // segment seg of walk block g's own region
            const int g = unit / NSEG, seg = unit % NSEG;
            nf = max(0, min(C.segcap, C.fill[g] - seg * C.segcap));
            c0 = (int64_t)g * C.cap + (int64_t)seg * C.segcap;
        } else {
            // a segment of the shared overflow pool
            const int64_t v0 = (int64_t)(unit - own_units) * C.segcap;
            nf = (int)max((int64_t)0, min((int64_t)C.segcap, no_all - v0));
            c0 = C.ovf_base + v0;
        }
        if (nf == 0) continue;
        my_base = bstart + C.counts[(int64_t)t * C.units + unit];
        const int nr = (nf + SC_CHUNKS - 1) / SC_CHUNKS;
        if (t == 0)
            for (int k = 0; k < SC_BUF && k < nr; ++k) issue(c0, nf, k, k);
        __syncthreads();
        for (int k = 0; k < nr; ++k) {
            const int b = k % SC_BUF;
            const bool ok = mbar_wait_bounded(&s.bar[b], (phase >> b) & 1u, SC_WAIT_LIMIT);
            if (ok) {
                phase ^= 1u << b;
                in_flight &= ~(1u << b);
            }
            if (__syncthreads_or(!ok)) {
                failed = true;
                break;
            }
            process(b, min(SC_CHUNKS, nf - k * SC_CHUNKS), c0, nf, k + SC_BUF < nr ? k + SC_BUF : -1);
        }
    }
    if (failed) {
        if (t == 0) {
            record_error(ctl, LRCC_ERR_TIMEOUT, -5);
            // let copies still in flight land before the block's shared memory goes away
            for (int b = 0; b < SC_BUF; ++b)
                if (in_flight & (1u << b)) mbar_wait_bounded(&s.bar[b], (phase >> b) & 1u, SC_WAIT_LIMIT);
        }
        __syncthreads();
    }
}

// Exercises the scatter's bounded wait on a barrier that no copy will ever
// complete: one arrival announces 16 bytes of transfer and no copy is issued,
// so the wait gives up after `polls` polls and records LRCC_ERR_TIMEOUT the
// way the scatter does. Nothing is in flight when the block exits.
__global__ void wait_check_kernel(DevCtl* ctl, int polls) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x != 0) return;
    mbar_init(&bar, 1);
    fence_proxy_async_smem();
    mbar_arrive_expect_tx(&bar, 16);
    if (!mbar_wait_bounded(&bar, 0, polls)) record_error(ctl, LRCC_ERR_TIMEOUT, -6);
}

}  // namespace

cudaError_t wait_check_enqueue(DevCtl* ctl, int polls, cudaStream_t s) {
    wait_check_kernel<<<1, 32, 0, s>>>(ctl, polls);
    return cudaGetLastError();
}

namespace {

// rank[element] from the pairs. Blocks take slices of PLACE_SLICE pairs from
// one counter in order, so at any moment the pairs in flight cover a few
// buckets and their rank writes stay in a window that L2 holds until every
// line is complete (a grid-stride loop would let blocks drift apart and
// spread the writes over far more memory than L2 holds).
// One block per SM and slices of 8192 pairs: the fewer pairs in flight, the
// narrower the window of rank lines the writes keep open in L2 (at 2^28:
// 1.37 ms, against 1.47 with two blocks per SM and 1.82 with 16384-pair slices).
#ifndef LRCC_PLACE_BLOCKS_PER_SM
#define LRCC_PLACE_BLOCKS_PER_SM 1
#endif
#ifndef LRCC_PLACE_SLICE_WARPS
#define LRCC_PLACE_SLICE_WARPS 32
#endif
constexpr int PLACE_SLICE = BLOCK * LRCC_PLACE_SLICE_WARPS;
__global__ void __launch_bounds__(BLOCK)
    rs_place(const uint64_t* __restrict__ pairs, int64_t n, int32_t* __restrict__ rank, DevCtl* ctl) {
    __shared__ int s_start;
    const int64_t m = min((int64_t)ctl->pairs, n);
    for (;;) {
        if (threadIdx.x == 0) s_start = atomicAdd(&ctl->place_next, PLACE_SLICE);
        __syncthreads();
        const int64_t start = s_start;
        __syncthreads();
        if (start >= m) break;
        const int64_t end = min(start + PLACE_SLICE, m);
        if (end - start == PLACE_SLICE) {
            // full slice: 2 U pairs per thread in flight
            constexpr int U = PLACE_SLICE / (2 * BLOCK) / 4;
            static_assert(U >= 1, "a slice holds at least 8 pairs per thread");
            for (int w = 0; w < 4; ++w) {
                ulonglong2 p[U];
#pragma unroll
                for (int u = 0; u < U; ++u)
                    p[u] = __ldcs(reinterpret_cast<const ulonglong2*>(pairs + start) + (w * U + u) * BLOCK + threadIdx.x);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    // ids come from the scatter and are < n; the checks only keep
                    // a corrupted pair from writing outside rank
                    if (lo32(p[u].x) < (uint64_t)n) rank[lo32(p[u].x)] = (int32_t)hi32(p[u].x);
                    if (lo32(p[u].y) < (uint64_t)n) rank[lo32(p[u].y)] = (int32_t)hi32(p[u].y);
                }
            }
        } else {
            for (int64_t i = start + threadIdx.x; i < end; i += BLOCK) {
                const uint64_t p = pairs[i];
                if (lo32(p) < (uint64_t)n) rank[lo32(p)] = (int32_t)hi32(p);
            }
        }
    }
}

// Expand at level >= 1: S[c] = S_next[owner] - prefix (RS5). Weighted ranks pass
// *chased, the elements the level's walks reached: all r of one list.
__global__ void __launch_bounds__(BLOCK)
    rs_expand(const uint64_t* __restrict__ P, uint32_t r, const int32_t* __restrict__ Snext, uint32_t rnext,
              int32_t* __restrict__ S, const unsigned long long* chased, DevCtl* ctl) {
    if (ctl->scan_bad) return;
    if (chased && blockIdx.x == 0 && threadIdx.x == 0 && *chased != r) record_error(ctl, LRCC_ERR_INVALID_INPUT, -3);
    for (uint32_t c = blockIdx.x * BLOCK + threadIdx.x; c < r; c += gridDim.x * BLOCK) {
        const uint64_t p = P[c];
        // an element no walk reached holds an old word: its owner is checked, so
        // that a malformed input can only give wrong values, never an access outside
        // Snext (it is recorded by the last level's total, or by the count above)
        S[c] = hi32(p) < rnext ? (int32_t)((uint32_t)Snext[hi32(p)] - lo32(p)) : 0;
    }
}

// Expand at level 0 into the caller's array: rank = S1[owner] - prefix - 1
// (bias 1); for weighted sums the inclusive suffix S1[owner] - prefix (bias 0).
template <bool VEC>
__global__ void __launch_bounds__(BLOCK)
    rs_expand0(const uint64_t* __restrict__ W, int64_t n, const int32_t* __restrict__ S1, int64_t r1,
               int32_t* __restrict__ rank, int bias, DevCtl* ctl) {
    if (ctl->scan_bad) return;
    const int64_t ngroups = (n + 3) >> 2;
    for (int64_t g = static_cast<int64_t>(blockIdx.x) * BLOCK + threadIdx.x; g < ngroups;
         g += static_cast<int64_t>(gridDim.x) * BLOCK) {
        const int64_t i0 = g * 4;
        uint64_t w[4];
        if (i0 + 3 < n) {
            const ulonglong2* s = reinterpret_cast<const ulonglong2*>(W + i0);
            const ulonglong2 a = __ldcs(s), b = __ldcs(s + 1);
            w[0] = a.x; w[1] = a.y; w[2] = b.x; w[3] = b.y;
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) w[q] = (i0 + q < n) ? W[i0 + q] : pack(SPL, 0);
        }
        int out[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t lo = lo32(w[q]), hi = hi32(w[q]);
            if ((lo & SPL) && hi < (uint64_t)r1) {
                out[q] = S1[hi] - bias;
            } else if (!(lo & SPL) && (hi & VIS) && (hi & ~VIS) < (uint64_t)r1) {
                out[q] = (int32_t)((uint32_t)S1[hi & ~VIS] - lo - (uint32_t)bias);
            } else {
                record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)(i0 + q));
                out[q] = -1;
            }
        }
        if (VEC && i0 + 3 < n) {
            __stcs(reinterpret_cast<int4*>(rank + i0), make_int4(out[0], out[1], out[2], out[3]));
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i0 + q < n) rank[i0 + q] = out[q];
        }
    }
}

// ------------------------------------------------ level 0, ranks in place
//
// First level of lists whose successors and ranks fit L2 together: the walk
// reads succ and writes one 4-byte record (owner, position) per element into
// the caller's rank array, which a streaming pass turns into the rank
// S1[owner] - 1 - position. No pass packs walk words first (splitters are
// recognised by their hashed offset), no workspace per element is needed, and
// 8 bytes per element are touched at random where the packed words cost 16;
// reading one array and writing another also keeps the walk from storing to
// lines it has just read (read-then-store runs at 29-65 G/s on GB300, reads
// alone at 290, stores alone at 180-206). lr_rank of 100,003 elements 67.7 ->
// 37.1 us, 2^20 106.7 -> 67.5, 15,000,001 479 -> 460 (there succ and rank are 120
// of L2's 129 MB, and the walk waits on HBM again).
//
// The record has the owner in its high bits and `pbits` bits of position. A
// sublist longer than 2^pbits goes on under an extra owner index nb + e, which
// the splitter before it links to; at most n >> pbits of them exist.

__global__ void __launch_bounds__(BLOCK)
    rs_walk_direct(const int32_t* __restrict__ succ, uint32_t* __restrict__ rec, Level0 L0, int pbits, int extras,
                   uint64_t* __restrict__ R1, DevCtl* ctl) {
    const Geo32 g = geo32(L0);
    uint32_t j = blockIdx.x * BLOCK + threadIdx.x;
    if (j >= g.nb) return;
    uint32_t cur = splitter_node32(j, g, nullptr), pos = 0;
    int32_t x = __ldg(succ + cur);
    CycleGuard guard(cur);
    uint32_t next = NIL;
    for (;;) {
        // cur belongs to owner j at position pos, x = succ[cur]
        rec[cur] = (j << pbits) | pos;
        ++pos;
        if (x == -1 || (uint32_t)x == cur) break;
        if ((uint32_t)x >= g.n || guard.seen((uint32_t)x)) {
            record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)cur);
            break;
        }
        cur = (uint32_t)x;
        x = __ldg(succ + cur);   // on its way while cur is tested
        const int sj = splitter_index32(cur, g);
        if (sj >= 0) {
            next = (uint32_t)sj;
            break;
        }
        if (pos >> pbits) {
            const int e = atomicAdd(&ctl->ff_extra, 1);
            if (e >= extras) {
                record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)cur);
                break;
            }
            R1[j] = pack(g.nb + (uint32_t)e, pos);
            j = g.nb + (uint32_t)e;
            pos = 0;
        }
    }
    R1[j] = pack(next, pos);
}

// Records -> ranks, in place. Records of elements no walk reached (a malformed
// input, which the last level has recorded) may name any owner: -1 then.
template <bool VEC>
__global__ void __launch_bounds__(BLOCK)
    rs_expand_direct(int32_t* rank, int64_t n, const int32_t* __restrict__ S1, uint32_t r1, int pbits) {
    const uint32_t mask = (1u << pbits) - 1;
    auto rank_of = [&](int32_t v) {
        const uint32_t o = (uint32_t)v >> pbits;
        return o < r1 ? S1[o] - 1 - (int32_t)((uint32_t)v & mask) : -1;
    };
    const int64_t ngroups = (n + 3) >> 2;
    for (int64_t g = static_cast<int64_t>(blockIdx.x) * BLOCK + threadIdx.x; g < ngroups;
         g += static_cast<int64_t>(gridDim.x) * BLOCK) {
        const int64_t i0 = g * 4;
        if (VEC && i0 + 3 < n) {
            int4* p = reinterpret_cast<int4*>(rank + i0);
            const int4 v = *p;
            *p = make_int4(rank_of(v.x), rank_of(v.y), rank_of(v.z), rank_of(v.w));
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i0 + q < n) rank[i0 + q] = rank_of(rank[i0 + q]);
        }
    }
}

// ------------------------------------------------ level 0, split arrays
//
// The paper's other first-level layout (Sec. 3.2, the "48 bit" version): the
// walk reads succ itself and keeps each element's ownership mark and local
// rank in two arrays, so a step reads succ[x] and mark[x] and writes mark[x]
// and lrank[x] (two random reads and two random writes, where the packed
// in-place word takes one of each). The mark is 16 bits while the level has
// fewer than 65,535 splitters (the paper's 2 + 4 bytes per element), 32 bits
// otherwise. A mark of all ones means "not visited"; a splitter's mark is its
// own index and its local rank 0.

template <typename MT>
__global__ void __launch_bounds__(BLOCK)
    rs_select0s(const int32_t* __restrict__ succ, MT* __restrict__ mark, int32_t* __restrict__ lrank,
                int32_t* __restrict__ snext, int32_t* __restrict__ sw, Level0 L0, DevCtl* ctl) {
    constexpr MT UNSEEN = MT(~MT(0));
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * BLOCK + threadIdx.x; i < L0.n;
         i += static_cast<int64_t>(gridDim.x) * BLOCK) {
        const int64_t j = splitter_index0(i, L0);
        mark[i] = j >= 0 ? (MT)j : UNSEEN;
        if (j >= 0) {
            const int v = succ[i];
            const bool tail = (v == -1) | (v == i);
            const bool bad = !tail && (v < 0 || v >= L0.n);
            if (bad) record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)i);
            snext[j] = (tail || bad) ? (int32_t)NIL : v;
            sw[j] = 1;
            lrank[i] = 0;
        }
    }
}

// Sublist walk over the split arrays; the hand-out of splitters to lanes is
// the same as rs_walk's. Output per splitter j: R1[j] = (next splitter,
// elements from j up to it), the packed words of level 1.
template <typename MT, int K>
__global__ void __launch_bounds__(BLOCK)
    rs_walk0s(const int32_t* __restrict__ succ, MT* __restrict__ mark, int32_t* __restrict__ lrank,
              const int32_t* __restrict__ snext, uint64_t* __restrict__ R1, int* work, Level0 L0, DevCtl* ctl) {
    constexpr MT UNSEEN = MT(~MT(0));
    constexpr int CHUNK = 64;
    const int r = (int)L0.nb;
    const int64_t n = L0.n;
    const int lane = threadIdx.x & 31;
    int pool = 0, pool_end = 0;
    bool exhausted = false;
    int j[K];
    uint32_t cur[K], pre[K];
    int64_t steps[K];
#pragma unroll
    for (int q = 0; q < K; ++q) {
        j[q] = -1;
        cur[q] = NIL;
        pre[q] = 0;
        steps[q] = 0;
    }
    for (;;) {
#pragma unroll
        for (int q = 0; q < K; ++q) {
            bool need = j[q] < 0;
            unsigned m = __ballot_sync(0xffffffffu, need);
            while (m && !exhausted) {
                if (pool >= pool_end) {
                    int b = 0;
                    if (lane == 0) b = atomicAdd(work, CHUNK);
                    b = __shfl_sync(0xffffffffu, b, 0);
                    if (b >= r) {
                        exhausted = true;
                        break;
                    }
                    pool = b;
                    pool_end = min(b + CHUNK, r);
                }
                const int avail = pool_end - pool;
                const int rk = __popc(m & lanemask_lt());
                if (need && rk < avail) {
                    const int jj = pool + rk;
                    j[q] = jj;
                    cur[q] = (uint32_t)snext[jj];
                    pre[q] = 1;
                    steps[q] = 0;
                    need = false;
                }
                pool += min(avail, __popc(m));
                m = __ballot_sync(0xffffffffu, need);
            }
        }
        bool act = false;
#pragma unroll
        for (int q = 0; q < K; ++q) act |= j[q] >= 0;
        if (!__any_sync(0xffffffffu, act)) break;
        MT mk[K];
        int sx[K];
#pragma unroll
        for (int q = 0; q < K; ++q) {
            const bool live = j[q] >= 0 && cur[q] < (uint32_t)n;
            mk[q] = live ? mark[cur[q]] : UNSEEN;
            sx[q] = live ? succ[cur[q]] : -1;
        }
#pragma unroll
        for (int q = 0; q < K; ++q) {
            if (j[q] < 0) continue;
            if (cur[q] == NIL) {
                R1[j[q]] = pack(NIL, pre[q]);
                j[q] = -1;
                continue;
            }
            if (cur[q] >= (uint32_t)n || ++steps[q] > n) {
                record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)cur[q]);
                R1[j[q]] = pack(NIL, pre[q]);
                j[q] = -1;
                continue;
            }
            if (mk[q] != UNSEEN) {
                // a splitter ends the sublist; any other marked element was
                // reached twice, so the input is not one list
                if (splitter_index0(cur[q], L0) == (int64_t)mk[q]) {
                    R1[j[q]] = pack((uint32_t)mk[q], pre[q]);
                } else {
                    record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)cur[q]);
                    R1[j[q]] = pack(NIL, pre[q]);
                }
                j[q] = -1;
                continue;
            }
            mark[cur[q]] = (MT)j[q];
            lrank[cur[q]] = (int32_t)pre[q];
            pre[q] += 1;
            const int v = sx[q];
            const bool tail = (v == -1) | ((uint32_t)v == cur[q]);
            const bool bad = !tail && (v < 0 || v >= n);
            if (bad) record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)cur[q]);
            cur[q] = (tail || bad) ? NIL : (uint32_t)v;
        }
    }
}

// rank = S1[mark] - lrank - 1 (RS5 over the split arrays).
template <typename MT>
__global__ void __launch_bounds__(BLOCK)
    rs_expand0s(const MT* __restrict__ mark, const int32_t* __restrict__ lrank, int64_t n,
                const int32_t* __restrict__ S1, int64_t r1, int32_t* __restrict__ rank, DevCtl* ctl) {
    constexpr MT UNSEEN = MT(~MT(0));
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * BLOCK + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * BLOCK) {
        const MT m = __ldcs(mark + i);
        if (m == UNSEEN || (int64_t)m >= r1) {
            // never visited: not reachable from the head
            record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)i);
            __stcs(rank + i, -1);
        } else {
            __stcs(rank + i, (int32_t)((uint32_t)S1[m] - (uint32_t)__ldcs(lrank + i) - 1u));
        }
    }
}

// ---------------------------------------------------------------- Wyllie

template <bool VEC>
__global__ void __launch_bounds__(BLOCK)
    wy_pack(const int32_t* __restrict__ succ, int64_t n, uint64_t* __restrict__ W, DevCtl* ctl) {
    const uint64_t pol = policy_evict_first();
    const int64_t ngroups = (n + 3) >> 2;
    for (int64_t g = static_cast<int64_t>(blockIdx.x) * BLOCK + threadIdx.x; g < ngroups;
         g += static_cast<int64_t>(gridDim.x) * BLOCK) {
        const int64_t i0 = g * 4;
        int s[4];
        if (VEC && i0 + 3 < n) {
            const int4 v = ld_stream_v4(succ + i0, pol);
            s[0] = v.x; s[1] = v.y; s[2] = v.z; s[3] = v.w;
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) s[q] = (i0 + q < n) ? succ[i0 + q] : -1;
        }
        uint64_t w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t i = i0 + q;
            const int v = s[q];
            const bool tail = (v == -1) | (v == i);
            const bool bad = !tail && (v < 0 || v >= n);
            if (i < n && bad) record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)i);
            // the tail points to itself with value 0, so jumps past it add nothing
            w[q] = (tail || bad) ? pack(0, (uint32_t)i) : pack(1, (uint32_t)v);
        }
        if (i0 + 3 < n) {
            ulonglong2* d = reinterpret_cast<ulonglong2*>(W + i0);
            d[0] = make_ulonglong2(w[0], w[1]);
            d[1] = make_ulonglong2(w[2], w[3]);
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i0 + q < n) W[i0 + q] = w[q];
        }
    }
}

// One pointer-jumping round: (r, s) <- (r + r[s], s[s]) from one 8-byte gather.
__global__ void __launch_bounds__(BLOCK)
    wy_jump(const uint64_t* __restrict__ Win, uint64_t* __restrict__ Wout, int64_t n) {
    const int64_t ngroups = (n + 3) >> 2;
    for (int64_t g = static_cast<int64_t>(blockIdx.x) * BLOCK + threadIdx.x; g < ngroups;
         g += static_cast<int64_t>(gridDim.x) * BLOCK) {
        const int64_t i0 = g * 4;
        uint64_t w[4], x[4];
        if (i0 + 3 < n) {
            const ulonglong2* s = reinterpret_cast<const ulonglong2*>(Win + i0);
            const ulonglong2 a = s[0], b = s[1];
            w[0] = a.x; w[1] = a.y; w[2] = b.x; w[3] = b.y;
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) w[q] = (i0 + q < n) ? Win[i0 + q] : 0ull;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = (i0 + q < n) ? Win[hi32(w[q])] : 0ull;
#pragma unroll
        for (int q = 0; q < 4; ++q) w[q] = pack(lo32(w[q]) + lo32(x[q]), hi32(x[q]));
        if (i0 + 3 < n) {
            ulonglong2* d = reinterpret_cast<ulonglong2*>(Wout + i0);
            d[0] = make_ulonglong2(w[0], w[1]);
            d[1] = make_ulonglong2(w[2], w[3]);
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i0 + q < n) Wout[i0 + q] = w[q];
        }
    }
}

// Last round writes the ranks; the head must reach the tail in n - 1 links.
template <bool VEC>
__global__ void __launch_bounds__(BLOCK)
    wy_final(const uint64_t* __restrict__ Win, int64_t n, int32_t head, int32_t* __restrict__ rank,
             DevCtl* ctl) {
    const int64_t ngroups = (n + 3) >> 2;
    for (int64_t g = static_cast<int64_t>(blockIdx.x) * BLOCK + threadIdx.x; g < ngroups;
         g += static_cast<int64_t>(gridDim.x) * BLOCK) {
        const int64_t i0 = g * 4;
        int out[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            out[q] = 0;
            if (i0 + q < n) {
                const uint64_t w = Win[i0 + q];
                const uint64_t x = Win[hi32(w)];
                out[q] = (int)(lo32(w) + lo32(x));
                if (i0 + q == head && out[q] != n - 1) record_error(ctl, LRCC_ERR_INVALID_INPUT, head);
            }
        }
        if (VEC && i0 + 3 < n) {
            *reinterpret_cast<int4*>(rank + i0) = make_int4(out[0], out[1], out[2], out[3]);
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i0 + q < n) rank[i0 + q] = out[q];
        }
    }
}

// ------------------------------------------------ batched lists as one list
//
// Lists k = 0..K-1 own elements [off[k], off[k+1]) with local ids. They are
// ranked as one list by the read-only first level: every element gets a
// global successor (off[k] + local, or -1 at a tail); the first non-empty
// list's head is the head; the head of every other list is a first-level
// splitter (its block's stratified splitter, or an extra splitter nb + e when
// that is another element); after the walk, the splitter that ends list k is
// linked to the head splitter of the next non-empty list, and the unused extra
// slots become a tail of empty splitters. Ranks along that one list are the
// local ranks plus the number of elements of the later lists, which are taken
// off the first-level splitters' suffix sums before the scatter. A walk never
// steps onto a head (nothing names it), so the walk recognises splitters by
// their hash as for one list.

// The list that holds element i (for empty lists, the last list starting at i).
__device__ __forceinline__ int64_t find_list(const int64_t* __restrict__ off, int64_t K, int64_t i) {
    int64_t lo = 0, hi = K - 1;
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (off[mid] <= i) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

constexpr int64_t LONG_LIST = int64_t(1) << 24;   // succ and rank of a longer one outgrow L2

// One block: the first list's head (head_dev[0]) and the head splitter of every
// list; head_dev[1] = the heads that became extra splitters, head_dev[2] = the
// elements of all lists, head_dev[3] and [4] = whether the read-only first level or
// the one with records in the rank array ranks them, head_dev[5] = the first list's
// length. Where the call left the form open (BATCH_EITHER) it is the read-only one
// when lists of more than LONG_LIST elements, which L2 does not hold, have most of
// the elements (one of 2^27 among 63 short ones: 4.5 ms, 8.3 with records; one of
// 2^26 and 63 of 2^20, a little over half: 3.5 and 4.1; one of 2^25 and 64 of 2^20, a third: 2.4
// with records, 2.7 read-only).
// The kernels after it trust the offsets, so they are checked here: from 0,
// non-decreasing, up to the n elements the call names (or, with pad_ok, ending
// before them). Others are reported and no form ranks the lists together (scan_bad).
__global__ void __launch_bounds__(1024)
    bl_heads(const int64_t* __restrict__ off, const int32_t* __restrict__ heads, int64_t K, int64_t n, int logD,
             int64_t nb, uint32_t seed, int32_t* __restrict__ head_spl, int32_t* __restrict__ extra_elem,
             int64_t* head_dev, int form, bool pad_ok, DevCtl* ctl) {
    __shared__ unsigned long long s_long;
    __shared__ int64_t s_first;
    __shared__ int s_warp[32];
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    bool ok = t != 32 || (off[0] == 0 && (off[K] == n || (pad_ok && off[K] < n)));
    if (t == 0) {
        s_long = 0;
        int64_t k0 = 0;
        while (k0 < K && off[k0 + 1] == off[k0]) ++k0;
        s_first = k0;
        int64_t gh = 0;
        if (k0 < K) {
            const int64_t len = off[k0 + 1] - off[k0];
            if (heads[k0] < 0 || heads[k0] >= len) record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)k0);
            else gh = off[k0] + heads[k0];
        }
        *head_dev = gh;
    }
    __syncthreads();
    const int64_t k0 = s_first;
    const int64_t gh0 = *head_dev;
    const int64_t D = int64_t(1) << logD;
    const int64_t bh = gh0 >> logD;
    const int64_t per = (K + 1023) / 1024;
    const int64_t kb = min(K, (int64_t)t * per), ke = min(K, kb + per);
    // a list's head and whether it is its block's stratified splitter
    auto head_of = [&](int64_t k, int64_t* gh, bool* strat) {
        const int64_t len = off[k + 1] - off[k];
        int64_t h = off[k];
        if (heads[k] < 0 || heads[k] >= len) record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)k);
        else h = off[k] + heads[k];
        const int64_t b = h >> logD;
        const uint32_t size = (uint32_t)min(D, n - (b << logD));
        *gh = h;
        *strat = b != bh && (uint32_t)(h - (b << logD)) == block_offset((uint32_t)b, size, seed);
    };
    int cnt = 0;
    unsigned long long in_long = 0;
    for (int64_t k = kb; k < ke; ++k) {
        const int64_t len = off[k + 1] - off[k];
        ok &= len >= 0;
        if (len > LONG_LIST) in_long += (unsigned long long)len;
        if (k == k0 || len == 0) continue;
        int64_t gh;
        bool strat;
        head_of(k, &gh, &strat);
        cnt += !strat;
    }
    if (in_long) atomicAdd(&s_long, in_long);
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    if (lane == 31) s_warp[wid] = incl;
    if (!__syncthreads_and(ok)) {   // (up to here the offsets were only counted with)
        if (t == 0) {
            record_error(ctl, LRCC_ERR_INVALID_INPUT, -9);
            ctl->scan_bad = 1;
            for (int i = 0; i < 6; ++i) head_dev[i] = 0;
        }
        return;
    }
    int before = 0, total = 0;
    for (int w = 0; w < 32; ++w) {
        before += w < wid ? s_warp[w] : 0;
        total += s_warp[w];
    }
    int e = before + incl - cnt;
    for (int64_t k = kb; k < ke; ++k) {
        if (off[k + 1] == off[k]) {
            head_spl[k] = -1;
            continue;
        }
        if (k == k0) {
            head_spl[k] = 0;
            continue;
        }
        int64_t gh;
        bool strat;
        head_of(k, &gh, &strat);
        if (strat) {
            const int64_t b = gh >> logD;
            head_spl[k] = (int32_t)(b >= bh ? b - bh : b - bh + nb);
        } else {
            head_spl[k] = (int32_t)(nb + e);
            extra_elem[e] = (int32_t)gh;
            ++e;
        }
    }
    if (t == 0) {
        ctl->ff_extra = total;
        head_dev[1] = total;
        head_dev[2] = off[K];
        const bool readonly = form == BATCH_READONLY || (form == BATCH_EITHER && 2 * s_long > (unsigned long long)n);
        head_dev[3] = readonly;
        head_dev[4] = !readonly;
        head_dev[5] = k0 < K ? off[k0 + 1] - off[k0] : 0;
    }
}

// What the read-only form of batched lists reads beside the walk's own arrays.
struct ListsGlobal {
    int32_t* gsucc;          // successors as global ids
    uint32_t* vis;           // the walk's marks and counts, to be cleared
    int* counts;
    int64_t ncounts;
};

// The read-only form's part of the first launch over the elements: block b's
// `tile` elements' successors as global ids, and its share of what has to be cleared.
template <int T>
__device__ void lists_to_global(const int32_t* __restrict__ succ, const int64_t* __restrict__ off, int64_t K, int64_t n,
                                int64_t tile, const ListsGlobal& G, DevCtl* ctl) {
    for (int64_t i = (int64_t)blockIdx.x * T + threadIdx.x; i < G.ncounts; i += (int64_t)gridDim.x * T) G.counts[i] = 0;
    const int64_t b = (int64_t)blockIdx.x * tile, e = min(n, b + tile);
    if (b >= e) return;
    for (int64_t w = (b >> 5) + threadIdx.x; w < (e + 31) >> 5; w += T) G.vis[w] = 0;   // tile: a multiple of 32
    const uint64_t pol = policy_evict_first();
    int64_t k = find_list(off, K, min(b + (int64_t)threadIdx.x, n - 1));
    constexpr int U = 8;   // loads in flight
    for (int64_t i0 = b + threadIdx.x; i0 < e; i0 += U * T) {
        int32_t sx[U];
#pragma unroll
        for (int q = 0; q < U; ++q) sx[q] = i0 + q * T < e ? ld_stream(succ + i0 + q * T, pol) : -1;
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const int64_t i = i0 + q * T;
            if (i >= e) break;
            while (off[k + 1] <= i) ++k;
            const int64_t base = off[k], len = off[k + 1] - base;
            int32_t g = -1;
            if (sx[q] != -1 && sx[q] != i - base) {
                if (sx[q] < 0 || sx[q] >= len) record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)i);
                else g = (int32_t)(base + sx[q]);
            }
            G.gsucc[i] = g;
        }
    }
}

// The next non-empty list after list k, or K, and the word of a splitter that ends
// list k with `pos` elements: on to that list's head, with that list's length taken
// off its weight, so that every sum from there back is list k's own. (The sum from the
// first list's head is then that list's length if and only if all lists' elements were
// met: the lengths taken off are those of all the others.)
__device__ __forceinline__ uint64_t list_end(const int64_t* __restrict__ off, int64_t K, const int32_t* __restrict__ head_spl,
                                             int64_t k, uint32_t pos) {
    for (++k; k < K && off[k + 1] == off[k];) ++k;
    return k < K ? pack((uint32_t)head_spl[k], pos - (uint32_t)(off[k + 1] - off[k])) : pack(NIL, pos);
}

// After the read-only walk, whose words of the last sublists name no next splitter.
// Runs in blocks of the launch that scans the walk's counts (blocks first ..).
__device__ void lists_link(uint64_t* __restrict__ R1, const int64_t* __restrict__ off, int64_t K,
                           const int32_t* __restrict__ head_spl, Level0 L0, int first) {
    const int64_t gh = *L0.head_dev;
    L0.bh = gh >> L0.logD;
    L0.head_off = (uint32_t)(gh - (L0.bh << L0.logD));
    const int64_t r_real = L0.nb + *L0.extra_count;
    const int64_t stride = (int64_t)(gridDim.x - first) * blockDim.x;
    for (int64_t j = (int64_t)(blockIdx.x - first) * blockDim.x + threadIdx.x; j < r_real; j += stride) {
        const uint64_t w = R1[j];
        if (lo32(w) != NIL) continue;
        R1[j] = list_end(off, K, head_spl, find_list(off, K, splitter_node0(j, L0)), hi32(w));
    }
}

__global__ void __launch_bounds__(SCAN_THREADS)
    bl_scan_link(int* counts, int G, int* totals, uint64_t* __restrict__ R1, const int64_t* __restrict__ off, int64_t K,
                 const int32_t* __restrict__ head_spl, Level0 L0) {
    const bool run = L0.head_dev[3];
    if (blockIdx.x >= NBK) {
        if (run) lists_link(R1, off, K, head_spl, L0, NBK);
    } else if (run) {
        scan_counts(counts, G, totals);
    } else if (threadIdx.x == 0) {   // nothing was walked
        totals[blockIdx.x] = 0;
    }
}

// The lists ranked together with their records in the rank array (as
// rs_walk_direct does for one list), for lists that L2 holds one after another:
// walkers take the splitters in id order, so those in flight stay in a few
// lists whose successors and records are in L2. The walk reads the local ids
// itself, and the splitter that ends a list is linked to the next list's head
// on the spot. 2048 lists of 2^8 to 2^20 elements: 3.30 ms, against 5.87 through
// global successors, chunks, scatter and placement; the walk (2.4 ms, 104 G
// steps/s) is bound by its L2 requests (2.6 per element), the expansion (0.73 ms)
// by one gather each. Fewer warps keep more of the lists in flight in L2: with 44
// registers 10 of 16 blocks fit an SM (EITHER: both forms in the kernel), 3.46 ms with
// 12, 3.65 with all. Without the other form 38 registers, 12 blocks (14 lists of 2^20:
// walk 155 us, 161 with all).
constexpr int LISTS_BLOCK = 128;   // short blocks: one lasts as long as its longest sublist
template <bool EITHER>
__global__ void __launch_bounds__(LISTS_BLOCK, 1)
    rs_walk_lists(const int32_t* __restrict__ succ, uint32_t* __restrict__ rec, Level0 L0,
                  const int64_t* __restrict__ off, int64_t K, const int32_t* __restrict__ head_spl, int pbits,
                  int extras, uint64_t* __restrict__ R1, ListsGlobal LG, DevCtl* ctl) {
    if (!L0.head_dev[4]) {
        if (EITHER && L0.head_dev[3]) lists_to_global<LISTS_BLOCK>(succ, off, K, L0.n, (int64_t)LISTS_BLOCK << L0.logD, LG, ctl);
        return;
    }
    const int64_t gh = L0.head_dev[0];
    L0.bh = gh >> L0.logD;
    L0.head_off = (uint32_t)(gh - (L0.bh << L0.logD));
    const Geo32 g = geo32(L0);
    uint32_t j = blockIdx.x * LISTS_BLOCK + threadIdx.x;
    if (j >= g.nb + (uint32_t)L0.head_dev[1]) return;
    uint32_t cur = splitter_node32(j, g, L0.extra), pos = 0;
    if (cur >= L0.head_dev[2]) {   // behind the last list
        R1[j] = pack(NIL, 0);
        return;
    }
    int64_t k = find_list(off, K, cur);
    const uint32_t base = (uint32_t)off[k], len = (uint32_t)(off[k + 1] - off[k]);
    int32_t x = __ldg(succ + cur);
    CycleGuard guard(cur);
    uint64_t last = NIL;   // the word's next splitter, and what goes off its weight
    for (;;) {
        // cur (a global id) belongs to owner j at position pos, x is its local successor
        rec[cur] = (j << pbits) | pos;
        ++pos;
        if (x == -1 || (uint32_t)x == cur - base) {
            last = list_end(off, K, head_spl, k, 0);   // on to the next list's head
            break;
        }
        if ((uint32_t)x >= len || guard.seen(base + (uint32_t)x)) {
            record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)cur);
            break;
        }
        cur = base + (uint32_t)x;
        x = __ldg(succ + cur);   // on its way while cur is tested
        const int sj = splitter_index32(cur, g);
        if (sj >= 0) {
            last = (uint32_t)sj;
            break;
        }
        if (pos >> pbits) {
            const int e = atomicAdd(&ctl->ff_extra, 1);
            if (e >= extras) {
                record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)cur);
                break;
            }
            R1[j] = pack(g.nb + (uint32_t)e, pos);
            j = g.nb + (uint32_t)e;
            pos = 0;
        }
    }
    R1[j] = pack(lo32(last), pos + hi32(last));
}

// Records -> local ranks, as rs_expand_direct (list_end makes the owners' sums the
// lists' own). Elements behind the last list are left alone.
//
// AGAIN: when an error was recorded, the blocks take the lists one by one instead,
// each in global memory (W: 8 bytes per element), so that a list that is none
// spoils only its own ranks. A kernel of its own after this one for it costs every
// call 4 to 6 us of 70 to 90.
constexpr int AGAIN_CAP = 256;   // splitters of a list ranked that way (L1 for the gathers, not speed there)
template <bool VEC, bool AGAIN>
__global__ void __launch_bounds__(BLOCK)
    rs_expand_lists(int32_t* rank, int64_t n, const int32_t* __restrict__ S1, uint32_t r1, int pbits,
                    const int64_t* __restrict__ off, int64_t K, const int64_t* __restrict__ head_dev,
                    const int32_t* __restrict__ succ, const int32_t* __restrict__ heads, uint64_t* W, uint32_t seed,
                    DevCtl* ctl) {
    const int failed = AGAIN ? ctl->failed : 0;
    const int64_t total = n;
    n = head_dev[4] ? min(n, head_dev[2]) : 0;   // 0: not ranked in this form
    const uint32_t mask = (1u << pbits) - 1;
    if constexpr (AGAIN) {
        if (failed) {
            __shared__ uint64_t s_words[AGAIN_CAP];
            __shared__ uint2 s_sub[2 * BLOCK];
            __shared__ int s_k, s_work;
            for (;;) {
                const int64_t k = take_instance(&s_k, &ctl->batch_next, K);
                if (k < 0) return;
                const int64_t b = off[k], len = off[k + 1] - b;
                if (len == 0) continue;
                if (!list_in_range(b, len, total) || (k == 0 && b != 0) || heads[k] < 0 || heads[k] >= len) {
                    if (threadIdx.x == 0) record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)k);
                    continue;
                }
                list_ruling_set<BLOCK, AGAIN_CAP>(succ + b, len, heads[k], rank + b, W + b, s_words, s_sub, &s_work,
                                                  seed ^ (uint32_t)k, 2, ctl);
            }
        }
    }
    auto rank_of = [&](int32_t v) {
        const uint32_t o = (uint32_t)v >> pbits;
        return o < r1 ? (int32_t)((uint32_t)S1[o] - 1u - ((uint32_t)v & mask)) : -1;
    };
    // a block takes one stretch of the elements: its owners stay in few lists
    const int64_t per = ((n + gridDim.x - 1) / gridDim.x + 4 * BLOCK - 1) / (4 * BLOCK) * (4 * BLOCK);
    const int64_t b = per * blockIdx.x, e = min(n, b + per);
    for (int64_t i = b + threadIdx.x * 4; i < e; i += 4 * BLOCK) {
        if (VEC && i + 3 < e) {
            int4* p = reinterpret_cast<int4*>(rank + i);
            const int4 v = __ldcs(p);
            __stcs(p, make_int4(rank_of(v.x), rank_of(v.y), rank_of(v.z), rank_of(v.w)));
        } else {
            for (int q = 0; q < 4; ++q)
                if (i + q < e) rank[i + q] = rank_of(rank[i + q]);
        }
    }
}

// ------------------------------------------- range check of the values

// Weighted ranks by the ruling set keep every partial sum in the 31-bit
// fields of the packed words, whose top bits are the splitter and visited
// flags: the values must be non-negative and their total below 2^31. This pass
// (one streaming read of val) checks both; when they do not hold, the later
// kernels of the call return at once and the call reports invalid input.
__global__ void __launch_bounds__(BLOCK)
    rs_scan_check(const int32_t* __restrict__ val, int64_t n, DevCtl* ctl) {
    const uint64_t pol = policy_evict_first();
    unsigned long long sum = 0;
    bool neg = false;
    for (int64_t i = (int64_t)blockIdx.x * BLOCK + threadIdx.x; i < n; i += (int64_t)gridDim.x * BLOCK) {
        const int32_t v = ld_stream(val + i, pol);
        neg |= v < 0;
        sum += (unsigned long long)(uint32_t)v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (__any_sync(0xffffffffu, neg) && (threadIdx.x & 31) == 0) ctl->scan_bad = 1;
    if ((threadIdx.x & 31) == 0 && sum) atomicAdd(&ctl->scan_total, sum);
}

__global__ void rs_scan_verdict(DevCtl* ctl) {
    if (ctl->scan_bad || ctl->scan_total >= (1ull << 31)) {
        ctl->scan_bad = 1;
        record_error(ctl, LRCC_ERR_INVALID_INPUT, -6);
    }
}

// ------------------------------------------- weighted ranks, separate records

// First level of weighted ranks: W[i] = (next or NIL, value) is read and
// P[i] = (prefix sum, owner) written, one thread per splitter, the splitters
// recognised by their hashed offset. Sums are plain 32-bit words (modulo 2^32):
// nothing is marked in them. For one list the geometry's head is the list's; a
// forest has the heads as extra splitters (L0.extra, after the stratified ones).
// P is an array of its own (APART) or W itself: when both outgrow L2 a record
// written where its word was read costs one line where two arrays cost two, while
// inside L2 a store to a line just read costs more than one elsewhere (see
// rs_chase). lr_scan: 10^6 elements 89 us apart against 119, 4 * 10^6 147 against
// 184, 15 * 10^6 841 against 491. The loads matter: apart, read-only ones (50,000
// elements: 35.5 us, 42 with plain loads); in place, past L1, where a plain load
// leaves the line that the store then hits (a forest of 10^7 elements: walk 227 us,
// 1676 with plain loads).
template <bool APART>
__global__ void __launch_bounds__(BLOCK)
    rs_walk_values(const uint64_t* W, uint64_t* P, Level0 L0, uint64_t* __restrict__ R1, DevCtl* ctl) {
    if (ctl->scan_bad) return;
    auto load = [](const uint64_t* p) {
        return APART ? (uint64_t)__ldg(reinterpret_cast<const unsigned long long*>(p)) : ld_cg_u64(p);
    };
    const Geo32 g = geo32(L0);
    const uint32_t r = g.nb + (L0.extra_count ? (uint32_t)*L0.extra_count : 0u);
    unsigned long long visited = 0;
    for (uint32_t j = blockIdx.x * BLOCK + threadIdx.x; j < r; j += gridDim.x * BLOCK) {
        uint32_t cur = splitter_node32(j, g, L0.extra);
        uint64_t w = load(W + cur);
        P[cur] = pack(0, j);
        uint32_t pre = hi32(w), steps = 1, next = NIL;
        CycleGuard guard(cur);
        cur = lo32(w);
        while (cur != NIL) {
            if (cur >= g.n || guard.seen(cur)) {
                record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)cur);
                break;
            }
            w = load(W + cur);
            const int sj = splitter_index32(cur, g);
            if (sj >= 0) {
                next = (uint32_t)sj;
                break;
            }
            P[cur] = pack(pre, j);
            pre += hi32(w);
            ++steps;
            cur = lo32(w);
        }
        R1[j] = pack(next, pre);
        visited += steps;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) visited += __shfl_xor_sync(0xffffffffu, visited, o);
    if ((threadIdx.x & 31) == 0 && visited) atomicAdd(&ctl->visited, visited);
}

// out = (owner's sum) - prefix. The sums are words S[o * stride + at].
template <bool VEC>
__global__ void __launch_bounds__(BLOCK)
    rs_expand_values(const uint64_t* __restrict__ P, int64_t n, const uint32_t* __restrict__ S, int stride, int at,
                     int64_t r, int32_t* __restrict__ out, DevCtl* ctl) {
    if (ctl->scan_bad) return;
    auto sum_of = [&](uint64_t p) {
        const uint32_t o = hi32(p);   // an element no walk reached (reported already) may name any owner
        return o < r ? (int32_t)(S[(int64_t)o * stride + at] - lo32(p)) : 0;
    };
    const int64_t ngroups = (n + 3) >> 2;
    for (int64_t g = static_cast<int64_t>(blockIdx.x) * BLOCK + threadIdx.x; g < ngroups;
         g += static_cast<int64_t>(gridDim.x) * BLOCK) {
        const int64_t i0 = g * 4;
        if (i0 + 3 < n) {
            const ulonglong2* s = reinterpret_cast<const ulonglong2*>(P + i0);
            const ulonglong2 a = __ldcs(s), b = __ldcs(s + 1);
            const int4 r4 = make_int4(sum_of(a.x), sum_of(a.y), sum_of(b.x), sum_of(b.y));
            if (VEC) {
                __stcs(reinterpret_cast<int4*>(out + i0), r4);
            } else {
                out[i0] = r4.x; out[i0 + 1] = r4.y; out[i0 + 2] = r4.z; out[i0 + 3] = r4.w;
            }
        } else {
            for (int64_t i = i0; i < n; ++i) out[i] = sum_of(P[i]);
        }
    }
}

// ------------------------------------------- weighted ranks of a forest

// A forest of lists has no single head. Its weighted ranks take the ruling
// set with every list head as an extra first-level splitter (the heads are the
// elements no successor names, found with one bit per element in a bitmap L2
// holds); the first level walks as for one list, and the splitters, a much
// smaller forest, are summed by pointer jumping (Sec. 3.1): words (next or NIL,
// value), rounds of (next, value) <- (next[next], value + value[next]), inside
// one launch that stops when no link is left. What makes the input invalid:
// an element named twice (more links than named elements), a cycle without a
// splitter (elements no walk reached), a cycle with one (links left after the
// last round).
__global__ void __launch_bounds__(BLOCK)
    ff_links(const int32_t* __restrict__ succ, int64_t n, uint32_t* has_pred, DevCtl* ctl) {
    const uint64_t pol = policy_evict_first();
    const int64_t stride = (int64_t)gridDim.x * BLOCK;
    unsigned long long links = 0;
    for (int64_t i0 = (int64_t)blockIdx.x * BLOCK + threadIdx.x; i0 < n; i0 += 4 * stride) {
        int32_t sx[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) sx[q] = i0 + q * stride < n ? ld_stream(succ + i0 + q * stride, pol) : -1;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t i = i0 + q * stride;
            if (i >= n || sx[q] == -1 || sx[q] == i) continue;
            if (sx[q] < 0 || sx[q] >= n) {
                record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)i);
                continue;
            }
            // no answer is waited for: elements named twice show in the count
            atomicOr(has_pred + (sx[q] >> 5), 1u << (sx[q] & 31));
            ++links;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) links += __shfl_xor_sync(0xffffffffu, links, o);
    if ((threadIdx.x & 31) == 0 && links) atomicAdd(&ctl->links, links);
}

// Walk words, and the heads that are not stratified splitters as extra ones
// (indices nb, nb + 1, ... in no particular order: one counter atomic per warp
// and iteration).
__global__ void __launch_bounds__(BLOCK)
    ff_select(const int32_t* __restrict__ succ, const int32_t* __restrict__ val, int64_t n,
              const uint32_t* __restrict__ has_pred, uint64_t* __restrict__ W, int32_t* __restrict__ extra, Level0 L0,
              DevCtl* ctl) {
    constexpr int U = 4;   // groups of 32 elements per warp and iteration
    const uint64_t pol = policy_evict_first();
    const Geo32 g = geo32(L0);
    const int lane = threadIdx.x & 31;
    unsigned long long named = 0;
    const int64_t warp = ((int64_t)blockIdx.x * BLOCK + threadIdx.x) >> 5, warps = (int64_t)gridDim.x * (BLOCK / 32);
    for (int64_t b = warp * 32 * U; b < n; b += warps * 32 * U) {
        int32_t sx[U], v[U];
        uint32_t pw[U];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const int64_t i = b + q * 32 + lane;
            sx[q] = i < n ? ld_stream(succ + i, pol) : -1;
            v[q] = i < n ? ld_stream(val + i, pol) : 0;
            pw[q] = b + q * 32 < n ? has_pred[(b >> 5) + q] : 0xFFFFFFFFu;
        }
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const int64_t i = b + q * 32 + lane;
            const bool in = i < n;
            if (b + q * 32 < n && lane == 0) named += __popc(pw[q]);
            const bool head = in && !(pw[q] >> lane & 1);
            const bool more = head && splitter_index32((uint32_t)i, g) < 0;
            const unsigned m = __ballot_sync(0xffffffffu, more);
            if (m) {
                int first = 0;
                if (lane == 0) first = atomicAdd(&ctl->ff_extra, __popc(m));
                first = __shfl_sync(0xffffffffu, first, 0);
                if (more) extra[first + __popc(m & lanemask_lt())] = (int32_t)i;
            }
            const bool tail = (sx[q] == -1) | (sx[q] == i) | (sx[q] < 0) | (sx[q] >= n);
            if (in) W[i] = pack(tail ? NIL : (uint32_t)sx[q], (uint32_t)v[q]);
        }
    }
    if (lane == 0 && named) atomicAdd(&ctl->named, named);
}

// The splitter forest's sums by pointer jumping in place: every word (next, sum
// up to next) is read and written whole, and a word that another block has
// already taken further only lengthens the jump, so no second buffer and no
// copying of finished words is needed. Rounds end when no link is left, where a
// launch per round had to make as many as the longest possible list needs.
//
// Jumping gathers every word in every round, from lines that other warps write,
// and slows with the number of words. From RULERS_MIN words on only one word of
// every four jumps, a ruler at a hashed place of its block: it first walks to the
// next ruler, and when the rulers have their sums every other word walks to its
// next ruler, both about four steps that only read. One list of 2^26 elements: 4.28
// ms, against 1.01 times a launch per round (4.23 to 4.53 from one machine to the
// next) with every word jumping (2^25: 1.99, 1.03 times 1.94 to 2.04). Below, the two walks cost
// more than the rounds they thin out (10M elements, 629,000 words: 434 us against
// 417; 2^20 elements, 135,000 words: 137 against 124).
constexpr int64_t RULERS_MIN = int64_t(1) << 20;
__device__ __forceinline__ int64_t ruler_of(int64_t b) { return (b << 2) + (mix32((uint32_t)b) & 3u); }
__device__ __forceinline__ bool is_ruler(uint32_t j) { return (mix32(j >> 2) & 3u) == (j & 3u); }

// The word w = R[i] taken along its list to the next ruler or the end.
__device__ __forceinline__ uint64_t to_ruler(const uint64_t* R, int64_t i, uint64_t w, int64_t r, DevCtl* ctl) {
    CycleGuard guard((uint32_t)i);
    while (lo32(w) < (uint64_t)r && !is_ruler(lo32(w))) {
        if (guard.seen(lo32(w))) {
            record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)i);
            break;
        }
        const uint64_t x = ld_cg_u64(R + lo32(w));
        w = pack(lo32(x), hi32(w) + hi32(x));
    }
    return w;
}

__global__ void __launch_bounds__(GANG_THREADS, 1)
    ff_rounds(uint64_t* R, int64_t n, int64_t nb, GangCtl* gc, DevCtl* ctl) {
    __shared__ int s_flag;
    Gang G{gc, &gc->arrived[0], (int)gridDim.x, (int)blockIdx.x, 0, ctl, &s_flag};
    const bool lead = blockIdx.x == 0 && threadIdx.x == 0;
    const int64_t r = nb + ctl->ff_extra;
    const int64_t stride = (int64_t)gridDim.x * GANG_THREADS;
    const int64_t t0 = (int64_t)blockIdx.x * GANG_THREADS + threadIdx.x;
    const bool rulers = r >= RULERS_MIN;
    const int64_t units = rulers ? (r + 3) >> 2 : r;   // words that jump
    if (lead && (ctl->links != ctl->named || ctl->visited != (unsigned long long)n))
        record_error(ctl, LRCC_ERR_INVALID_INPUT, -7);
    if (rulers) {
        // only rulers are written and only other words are read
        for (int64_t b = t0; b < units; b += stride) {
            const int64_t i = ruler_of(b);
            if (i < r) R[i] = to_ruler(R, i, ld_cg_u64(R + i), r, ctl);
        }
        if (!G.sync()) return;
    }
    int cap = 2;
    while ((int64_t(1) << (cap - 2)) < r) ++cap;
    // false when a barrier gave up or the links do not end
    auto rounds = [&](auto at) {
        for (int round = 0;; ++round) {
            bool any = false;
            for (int64_t b0 = t0; b0 < units; b0 += 4 * stride) {
                int64_t i[4];
                uint64_t w[4], x[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    i[q] = b0 + q * stride < units ? at(b0 + q * stride) : r;
                    w[q] = i[q] < r ? ld_cg_u64(R + i[q]) : pack(NIL, 0);
                }
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    x[q] = lo32(w[q]) < (uint64_t)r ? ld_cg_u64(R + lo32(w[q])) : pack(NIL, 0);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (lo32(w[q]) == NIL) continue;
                    R[i[q]] = pack(lo32(x[q]), hi32(w[q]) + hi32(x[q]));
                    any |= lo32(x[q]) != NIL;
                }
            }
            if (__syncthreads_or(any) && threadIdx.x == 0) atomicAdd(&gc->kept[round % 3], 1ull);
            if (lead) gc->kept[(round + 1) % 3] = 0;
            if (!G.sync()) return false;
            const bool more = *reinterpret_cast<volatile unsigned long long*>(&gc->kept[round % 3]) != 0;
            if (!more || round >= cap) {
                if (lead) {
                    if (more) record_error(ctl, LRCC_ERR_INVALID_INPUT, -2);
                    ctl->jump_rounds = round + 1;
                }
                return !more;
            }
        }
    };
    if (!rulers) {
        rounds([](int64_t b) { return b; });
        return;
    }
    if (!rounds([](int64_t b) { return ruler_of(b); })) return;
    // the other words: to their ruler, whose word now reaches the end (a word met
    // on the way may be finished already, which ends the walk there)
    for (int64_t i = t0; i < r; i += stride) {
        if (is_ruler((uint32_t)i)) continue;
        uint64_t w = ld_cg_u64(R + i);
        if (lo32(w) == NIL) continue;
        w = to_ruler(R, i, w, r, ctl);
        if (lo32(w) < (uint64_t)r && is_ruler(lo32(w))) {
            const uint64_t x = ld_cg_u64(R + lo32(w));
            w = pack(lo32(x), hi32(w) + hi32(x));
        }
        R[i] = w;
    }
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

lrcc_status launch_small(Ctx* c, cudaStream_t s, const int32_t* succ, int n, int head, int32_t* rank, uint32_t seed,
                         const int32_t* val = nullptr) {
    const size_t smem = br_smem(n);
    allow_smem(c, (const void*)lr_small_kernel, br_smem(16384));
    phase_begin(c, s);
    lr_small_kernel<<<1, FINAL_THREADS, smem, s>>>(succ, val, n, head, rank, seed, c->ctl);
    phase_end(c, s, PH_SMALL);
    return cuda_status(cudaGetLastError());
}

lrcc_status launch_small_wyllie(Ctx* c, cudaStream_t s, const int32_t* succ, int n, int head, int32_t* rank) {
    const int per = n <= 4096 ? 4 : (n <= 8192 ? 8 : 16);
    const size_t smem = 2 * sizeof(int) * per * FINAL_THREADS;
    const void* k = per == 4 ? (const void*)wy_small_kernel<4>
                  : per == 8 ? (const void*)wy_small_kernel<8> : (const void*)wy_small_kernel<16>;
    allow_smem(c, k, smem);
    phase_begin(c, s);
    if (per == 4) wy_small_kernel<4><<<1, FINAL_THREADS, smem, s>>>(succ, n, head, rank, c->ctl);
    else if (per == 8) wy_small_kernel<8><<<1, FINAL_THREADS, smem, s>>>(succ, n, head, rank, c->ctl);
    else wy_small_kernel<16><<<1, FINAL_THREADS, smem, s>>>(succ, n, head, rank, c->ctl);
    phase_end(c, s, PH_SMALL);
    return cuda_status(cudaGetLastError());
}

int stream_grid(Ctx* c, int64_t groups, const void* kernel) {
    const int pg = persistent_grid(c, kernel, BLOCK);
    const int64_t need = (groups + BLOCK - 1) / BLOCK;
    return (int)std::max<int64_t>(1, std::min<int64_t>(need, pg));
}

// Weighted ranks up to this size keep their records apart from the walk words
// (16 bytes per element, within L2 up to about here).
constexpr int64_t WALK_NEAR = int64_t(1) << 22;

void enqueue_expand_values(Ctx* c, cudaStream_t s, const uint64_t* P, int64_t n, const uint32_t* S, int stride, int at,
                           int64_t r, int32_t* out) {
    const bool v = aligned16(out);
    const void* k = v ? (const void*)rs_expand_values<true> : (const void*)rs_expand_values<false>;
    const int g = stream_grid(c, (n + 3) / 4, k);
    phase_begin(c, s);
    if (v) rs_expand_values<true><<<g, BLOCK, 0, s>>>(P, n, S, stride, at, r, out, c->ctl);
    else rs_expand_values<false><<<g, BLOCK, 0, s>>>(P, n, S, stride, at, r, out, c->ctl);
    phase_end(c, s, PH_EXPAND0);
}

}  // namespace

// --------------------------------------------------------------- planning

lrcc_status rs_chase_probe_run(Ctx* c, const int32_t* succ, int64_t n, int64_t chains, int64_t steps,
                               int64_t* out) {
    cudaMemsetAsync(out, 0, sizeof(int64_t), c->stream);
    const int64_t threads = (chains + PROBE_K - 1) / PROBE_K;
    const int64_t g = (threads + BLOCK - 1) / BLOCK;
    rs_chase_probe<<<(unsigned)g, BLOCK, 0, c->stream>>>(succ, n, chains, steps,
                                                         reinterpret_cast<unsigned long long*>(out));
    return cuda_status(cudaGetLastError());
}

int rs_walk_grid(Ctx* c, const Plan& p) {
    const void* k = p.rs_chains >= 4 ? (const void*)rs_walk0c<4>
                  : p.rs_chains == 2 ? (const void*)rs_walk0c<2> : (const void*)rs_walk0c<1>;
    return persistent_grid(c, k, BLOCK);
}

int rs_walk_grid_current(const Plan& p) {
    int dev = 0, sms = 0, per_sm = 0;
    const void* k = p.rs_chains >= 4 ? (const void*)rs_walk0c<4>
                  : p.rs_chains == 2 ? (const void*)rs_walk0c<2> : (const void*)rs_walk0c<1>;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, BLOCK, 0) != cudaSuccess || per_sm < 1 ||
        sms < 1) {
        cudaGetLastError();
        return 152 * 8;
    }
    return per_sm * sms;
}

RsLayout rs_layout(int64_t n, const Plan& p, int walk_grid, int64_t extra1, int64_t given1, bool direct, bool values) {
    RsLayout L;
    values = values && p.rs_level0 == 1 && n > p.rs_small && n <= WALK_NEAR;
    L.values = values;
    L.size[0] = n;
    // (batched lists, extra1 > 0, stay in L2 one after another at any total)
    direct = direct && n > p.rs_small && (extra1 > 0 || (p.rs_level0 == 1 && n <= DIRECT_MAX));
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off = align_up(off + bytes, 256);
        return o;
    };
    // in-place walk words, the (element, rank) pairs of the read-only walk, or
    // the split mark and local-rank arrays (each 256-byte aligned)
    if (!direct || p.rs_level0 == 2) L.off_W0 = take(sizeof(uint64_t) * (size_t)n + 256);
    if (values) L.off_P0 = take(sizeof(uint64_t) * (size_t)n);
    int64_t cur = n;
    int lvl = 0;
    while (cur > p.rs_small && lvl < MAX_LEVELS) {
        // spacing: a power of two, at least 4 (one block holds whole 4-element groups)
        int64_t spacing = lvl == 0 ? p.rs_spacing0 : p.rs_spacing;
        int logD = 2;
        while (logD < 20 && (int64_t(1) << (logD + 1)) <= spacing) ++logD;
        if (lvl == MAX_LEVELS - 1)  // last allowed level must fit one block
            while (logD < 30 && ((cur + (int64_t(1) << logD) - 1) >> logD) > p.rs_small) ++logD;
        // level 1 may hold extra splitters (the heads of batched lists ranked as one list)
        int64_t nb = ((cur + (int64_t(1) << logD) - 1) >> logD) + (lvl == 0 ? extra1 : 0);
        if (lvl == 0 && given1 > 0) nb = given1;   // first-level splitters chosen by the caller
        if (lvl == 0 && (direct || extra1 > 0)) L.fixed = nb - extra1;
        if (lvl == 0 && direct) {
            // as many position bits as the owners leave, extra owners included
            const int64_t heads = nb;   // with the heads of batched lists
            L.direct = true;
            for (L.pbits = 31; L.pbits > 0; --L.pbits) {
                nb = heads + (n >> L.pbits);
                if (nb <= (int64_t(1) << (32 - L.pbits))) break;
            }
        }
        L.logD[lvl] = logD;
        ++lvl;
        L.size[lvl] = nb;
        L.off_R[lvl] = take(sizeof(uint64_t) * (size_t)nb);
        if (lvl == 1 && !direct && !values) {
            L.off_snext = take(sizeof(int32_t) * (size_t)nb);
            L.off_sw = take(sizeof(int32_t) * (size_t)nb);
        }
        L.off_S[lvl] = take(sizeof(int32_t) * (size_t)nb);
        cur = nb;
    }
    L.levels = lvl;
    // level 1's records take over the successors and weights, which only the first level's walk reads
    for (int l = 1; l < lvl; ++l)
        L.off_P[l] = l == 1 && !direct && !values ? L.off_snext : take(sizeof(uint64_t) * (size_t)L.size[l]);
    L.readonly = p.rs_level0 == 2 && lvl > 0 && walk_grid > 0;
    L.split = p.rs_level0 == 3 && lvl > 0;
    if (L.readonly) {
        const int64_t G = walk_grid;
        L.grid = G;
        // own region per block: its share of the elements in chunks of 8, plus
        // the padding of its share of the sublists, with 30 % slack
        L.cap = (int64_t)(1.1 * (double)n / (double)G / CIDS + 0.6 * (double)L.size[1] / (double)G) + 16;
        // NSEG segments of an even number of chunks, so every segment's headers
        // start 16-byte aligned (bulk copies)
        L.segcap = (int)((L.cap + 2 * NSEG - 1) / (2 * NSEG)) * 2;
        L.cap = (int64_t)L.segcap * NSEG;
        // the shared pool alone can hold every chunk of a valid list (at most
        // n/8 full chunks plus one partial chunk per sublist), however unevenly
        // the sublists fall on the blocks
        L.ovf_cap = n / CIDS + L.size[1] + 1024;
        L.ovf_cap += L.ovf_cap & 1;
        L.units = (int)(G * NSEG + (L.ovf_cap + L.segcap - 1) / L.segcap);
        const int64_t chunks = G * L.cap + L.ovf_cap;
        L.off_ids = take(sizeof(int32_t) * CIDS * (size_t)chunks);
        L.off_meta = take(sizeof(uint64_t) * (size_t)chunks);
        L.off_fill = take(sizeof(int) * (size_t)G);
        L.off_counts = take(sizeof(int) * (size_t)NBK * (size_t)L.units);
        L.off_totals = take(sizeof(int) * (size_t)NBK);
        L.off_vis = take(sizeof(uint32_t) * (size_t)((n + 31) / 32));
    }
    L.bytes = off;
    return L;
}

// Batched lists ranked together as one list: whether, the plan, the layout and
// the workspace. One block ranks a list of up to 24,576 elements in some 30 us
// and needs 270 us and more for a longer one, where the whole GPU takes 60 to 100
// for all of them; the host only knows the total and the count, so the mean
// decides: lists of 2^12 elements on average go together (16 lists of up to 2^17:
// 62 us, 269 by blocks; 64 of up to 2^20: 166 against 2618), of 2^13 when they
// total less than 2^17, shorter ones by blocks (2000 of up to 2^14: 83 us). A total
// above 2^24 is never left to single blocks, where one long list among many short
// ones lasts as long as it does alone (5000 lists of 256 elements and one of 2^24: 64.7
// ms by blocks, 0.67 together), although short lists alone are faster
// there (12,000 of 1500: 232 us by blocks, 323 together). Lists of 2^22
// elements and less on average keep their records in the rank array, longer ones (and
// those ranked in place) outgrow L2 and take the read-only first level (chunks,
// scatter, placement) above 2^24 in all (3 lists of 2^23: 858 us, 40.7 ms by blocks).
// The mean says little where a few long lists have most of the elements: from 2^25 on,
// where a list can outgrow L2, the device chooses between the two (bl_heads); the
// launches of the other one end at once (16 us of 735 for 40 lists of 2^20).
constexpr int64_t UNION_MIN = int64_t(1) << 15;
constexpr int64_t UNION_DIRECT_MEAN = int64_t(1) << 22;
constexpr int64_t UNION_LARGE = int64_t(1) << 24;
constexpr int64_t UNION_EITHER_MIN = int64_t(1) << 25;
constexpr int64_t UNION_MAX = int64_t(0x7FFFFFFE);   // global ids are int32

BatchMode lr_batch_mode(int64_t total, int64_t K, const Plan& batch_plan, bool overlap) {
    if (batch_plan.rs_level0 != 2 || total < UNION_MIN || total > UNION_MAX - K) return BATCH_BLOCKS;
    const int64_t min_mean = int64_t(1) << (total < (int64_t(1) << 17) ? 13 : 12);
    if (total <= UNION_DIRECT_MEAN * K && !overlap)
        return total >= UNION_EITHER_MIN                        ? BATCH_EITHER
               : total >= min_mean * K || total > UNION_LARGE ? BATCH_DIRECT
                                                              : BATCH_BLOCKS;
    return total > UNION_LARGE ? BATCH_READONLY : BATCH_BLOCKS;
}

// Up to this total the lists are ranked one by one when that fails together (one of
// them is none), and elements may follow the last; a larger total keeps no room for it.
constexpr int64_t UNION_AGAIN_MAX = UNION_LARGE;

struct UnionPlan {
    Plan p;
    bool again;
    RsLayout L;
    size_t off_gsucc, off_head_spl, off_extra, off_head_dev, bytes;
};

UnionPlan union_plan(int walk_grid, int64_t total, int64_t K, BatchMode mode) {
    UnionPlan U;
    const bool direct = mode != BATCH_READONLY;
    U.p = plan_for(KIND_LR, total);
    U.p.rs_level0 = mode == BATCH_DIRECT ? 1 : 2;
    U.p.rs_small = std::min(U.p.rs_small, 16384);
    U.L = rs_layout(total, U.p, walk_grid, K, 0, direct);
    size_t off = align_up(U.L.bytes, 256);
    U.off_gsucc = off;
    if (mode != BATCH_DIRECT) off = align_up(off + sizeof(int32_t) * (size_t)total, 256);
    U.off_head_spl = off;
    off = align_up(off + sizeof(int32_t) * (size_t)K, 256);
    U.off_extra = off;
    off = align_up(off + sizeof(int32_t) * (size_t)K, 256);
    U.again = direct && total <= UNION_AGAIN_MAX;
    // (the words of lists ranked one by one lie in front: blocks that start later still read it)
    if (U.again) off = std::max(off, align_up(sizeof(uint64_t) * (size_t)total, 256));
    U.off_head_dev = off;
    U.bytes = off + 256;
    return U;
}

size_t lr_batched_union_ws(int walk_grid, int64_t total, int64_t K, BatchMode mode) {
    return union_plan(walk_grid, total, K, mode).bytes;
}

lrcc_status lr_batched_union(Ctx* c, cudaStream_t s, const int32_t* succ, const int64_t* off, const int32_t* heads,
                             int64_t K, int64_t total, int32_t* rank, BatchMode mode) {
    const UnionPlan P = union_plan(rs_walk_grid(c, plan_for(KIND_LR, total)), total, K, mode);
    if (!(P.L.readonly || P.L.direct) || P.L.levels == 0 || c->ws_bytes < P.bytes) return LRCC_ERR_ARG;
    char* base = static_cast<char*>(c->ws);
    BatchUnion U;
    U.off = off;
    U.heads = heads;
    U.K = K;
    U.gsucc = reinterpret_cast<int32_t*>(base + P.off_gsucc);
    U.head_spl = reinterpret_cast<int32_t*>(base + P.off_head_spl);
    U.extra_elem = reinterpret_cast<int32_t*>(base + P.off_extra);
    U.head_dev = reinterpret_cast<int64_t*>(base + P.off_head_dev);
    U.form = mode;
    U.again = P.again;
    return lr_enqueue_rs(c, s, succ, total, 0, rank, P.p, P.L, nullptr, &U);
}

size_t lr_wyllie_ws(int64_t n, const Plan&) { return 2 * align_up(sizeof(uint64_t) * (size_t)n, 256); }

// ------------------------------------------------------------ enqueueing

lrcc_status lr_enqueue_rs(Ctx* c, cudaStream_t s, const int32_t* succ, int64_t n, int32_t head,
                          int32_t* rank, const Plan& p, const RsLayout& L, const int32_t* val,
                          const BatchUnion* U, const int32_t* given, int64_t given_r) {
    // caller-chosen first-level splitters need the in-place first level
    if (given && (L.readonly || L.split || L.direct || U)) return LRCC_ERR_ARG;
    // batched lists ranked as one list need the read-only first level or records in the rank array
    if (U && (!(L.readonly || L.direct) || val)) return LRCC_ERR_ARG;
    // weighted sums use the in-place first level (the others count positions)
    if (val && (L.readonly || L.split || L.direct)) return LRCC_ERR_ARG;
    if (val) {
        phase_begin(c, s);
        rs_scan_check<<<stream_grid(c, n, (const void*)rs_scan_check), BLOCK, 0, s>>>(val, n, c->ctl);
        rs_scan_verdict<<<1, 1, 0, s>>>(c->ctl);
        phase_end(c, s, PH_SELECT0);
    }
    if (n <= p.rs_small || L.levels == 0) return launch_small(c, s, succ, (int)n, head, rank, (uint32_t)p.seed, val);
    char* base = static_cast<char*>(c->ws);
    auto R = [&](int l) { return reinterpret_cast<uint64_t*>(base + L.off_R[l]); };
    auto P = [&](int l) { return reinterpret_cast<uint64_t*>(base + L.off_P[l]); };
    int32_t* SN = reinterpret_cast<int32_t*>(base + L.off_snext);
    int32_t* SW = reinterpret_cast<int32_t*>(base + L.off_sw);
    auto S = [&](int l) { return reinterpret_cast<int32_t*>(base + L.off_S[l]); };
    uint64_t* W0 = reinterpret_cast<uint64_t*>(base + L.off_W0);
    DevCtl* ctl = c->ctl;
    const uint32_t seed0 = (uint32_t)(p.seed ^ (p.seed >> 32));

    // level 0
    const bool vec = aligned16(succ) && (!val || aligned16(val));
    const int64_t groups = (n + 3) / 4;
    if (!L.readonly && !L.split && !L.direct) {
        const void* k = vec ? (const void*)rs_select0<true> : (const void*)rs_select0<false>;
        const int g = stream_grid(c, groups, k);
        phase_begin(c, s);
        if (vec)
            rs_select0<true><<<g, BLOCK, 0, s>>>(succ, val, n, head, W0, SN, SW, L.logD[0], L.size[1],
                                                 seed0, ctl, given == nullptr && !L.values);
        else
            rs_select0<false><<<g, BLOCK, 0, s>>>(succ, val, n, head, W0, SN, SW, L.logD[0], L.size[1],
                                                  seed0, ctl, given == nullptr && !L.values);
        if (given) {
            const int gm = stream_grid(c, given_r, (const void*)rs_mark_given);
            rs_mark_given<<<gm, BLOCK, 0, s>>>(W0, n, head, given, given_r, SN, SW, ctl);
        }
        phase_end(c, s, PH_SELECT0);
    }
    Level0 L0;
    L0.n = n;
    L0.logD = L.logD[0];
    L0.nb = (n + (int64_t(1) << L0.logD) - 1) >> L0.logD;   // stratified splitters (level 1 may hold more)
    L0.bh = (int64_t)head >> L0.logD;
    L0.head_off = (uint32_t)(head - (L0.bh << L0.logD));
    L0.seed = seed0;
    if (U) {
        phase_begin(c, s);
        bl_heads<<<1, 1024, 0, s>>>(U->off, U->heads, U->K, n, L0.logD, L0.nb, seed0, U->head_spl, U->extra_elem,
                                    U->head_dev, U->form, U->again, ctl);
        phase_end(c, s, PH_BATCH_PREP);
        L0.head_dev = U->head_dev;
        L0.extra = U->extra_elem;
        L0.extra_count = &ctl->ff_extra;
    }
    // split arrays: 16-bit marks while every splitter index fits below the
    // all-ones "not visited" value
    const bool mark16 = L.size[1] < 0xFFFF;
    void* mark = base + L.off_W0;
    int32_t* lrank = reinterpret_cast<int32_t*>(
        base + L.off_W0 + align_up((mark16 ? sizeof(uint16_t) : sizeof(uint32_t)) * (size_t)n, 256));
    if (L.split) {
        phase_begin(c, s);
        if (mark16) {
            const int g = stream_grid(c, n, (const void*)rs_select0s<uint16_t>);
            rs_select0s<uint16_t><<<g, BLOCK, 0, s>>>(succ, (uint16_t*)mark, lrank, SN, SW, L0, ctl);
        } else {
            const int g = stream_grid(c, n, (const void*)rs_select0s<uint32_t>);
            rs_select0s<uint32_t><<<g, BLOCK, 0, s>>>(succ, (uint32_t*)mark, lrank, SN, SW, L0, ctl);
        }
        phase_end(c, s, PH_SELECT0);
    }
    Chunks C;
    C.ids = reinterpret_cast<int32_t*>(base + L.off_ids);
    C.meta = reinterpret_cast<uint64_t*>(base + L.off_meta);
    C.fill = reinterpret_cast<int*>(base + L.off_fill);
    C.counts = reinterpret_cast<int*>(base + L.off_counts);
    C.totals = reinterpret_cast<int*>(base + L.off_totals);
    C.vis = reinterpret_cast<uint32_t*>(base + L.off_vis);
    C.cap = L.cap;
    C.segcap = L.segcap;
    C.units = L.units;
    C.ovf_cap = L.ovf_cap;
    C.ovf_base = L.grid * L.cap;
    int lg = 0;
    while ((int64_t(1) << lg) < n) ++lg;
    C.shift = std::max(0, lg - NBK_LOG);
    C.careful = int64_t(32) << L.logD[0];
    auto walk0 = [&] {
        const int r = (int)L.size[1];
        int* work = &ctl->work[0];
        phase_begin(c, s);
        if (p.rs_chains >= 4) {
            const int g = persistent_grid(c, (const void*)rs_walk<4>, BLOCK);
            rs_walk<4><<<g, BLOCK, 0, s>>>(W0, SN, SW, R(1), r, work, n, ctl);
        } else if (p.rs_chains == 2) {
            const int g = persistent_grid(c, (const void*)rs_walk<2>, BLOCK);
            rs_walk<2><<<g, BLOCK, 0, s>>>(W0, SN, SW, R(1), r, work, n, ctl);
        } else {
            const int g = persistent_grid(c, (const void*)rs_walk<1>, BLOCK);
            rs_walk<1><<<g, BLOCK, 0, s>>>(W0, SN, SW, R(1), r, work, n, ctl);
        }
        phase_end(c, s, PH_WALK0);
    };
    // overflow units' counts are accumulated with atomics (own units are stored whole)
    const int64_t ncounts = (int64_t)NBK * L.units;
    if (U) {
        // the walk over the lists, or the global successors of the read-only one
        phase_begin(c, s);
        auto walk = L.readonly ? rs_walk_lists<true> : rs_walk_lists<false>;
        walk<<<(unsigned)((L0.nb + U->K + LISTS_BLOCK - 1) / LISTS_BLOCK), LISTS_BLOCK, 0, s>>>(
            succ, reinterpret_cast<uint32_t*>(rank), L0, U->off, U->K, U->head_spl, L.pbits, (int)(L.size[1] - L.fixed),
            R(1), ListsGlobal{U->gsucc, C.vis, C.counts, L.readonly ? ncounts : 0}, ctl);
        phase_end(c, s, L.direct ? PH_WALK0 : PH_BATCH_PREP);
    }
    if (L.readonly) {
        if (!U) {
            cudaMemsetAsync(C.vis, 0, sizeof(uint32_t) * (size_t)((n + 31) / 32), s);
            cudaMemsetAsync(C.counts, 0, sizeof(int) * (size_t)ncounts, s);
        }
        const int32_t* next = U ? U->gsucc : succ;
        const int G = (int)L.grid;
        phase_begin(c, s);
        if (p.rs_chains >= 4) rs_walk0c<4><<<G, BLOCK, 0, s>>>(next, L0, C, R(1), &ctl->work[0], ctl);
        else if (p.rs_chains == 2) rs_walk0c<2><<<G, BLOCK, 0, s>>>(next, L0, C, R(1), &ctl->work[0], ctl);
        else rs_walk0c<1><<<G, BLOCK, 0, s>>>(next, L0, C, R(1), &ctl->work[0], ctl);
        phase_end(c, s, PH_WALK0);
        phase_begin(c, s);
        if (U)
            bl_scan_link<<<NBK + 4 * c->sms, SCAN_THREADS, 0, s>>>(C.counts, L.units, C.totals, R(1), U->off, U->K,
                                                                  U->head_spl, L0);
        else
            rs_scan_counts<<<NBK, SCAN_THREADS, 0, s>>>(C.counts, L.units, C.totals);
        phase_end(c, s, PH_SCAN);
    } else if (L.split) {
        auto walk0s = [&](auto mt, auto k) {
            using MT = decltype(mt);
            constexpr int K = decltype(k)::value;
            const int g = persistent_grid(c, (const void*)rs_walk0s<MT, K>, BLOCK);
            rs_walk0s<MT, K><<<g, BLOCK, 0, s>>>(succ, (MT*)mark, lrank, SN, R(1), &ctl->work[0], L0, ctl);
        };
        phase_begin(c, s);
        if (mark16) {
            if (p.rs_chains >= 4) walk0s(uint16_t(), std::integral_constant<int, 4>());
            else if (p.rs_chains == 2) walk0s(uint16_t(), std::integral_constant<int, 2>());
            else walk0s(uint16_t(), std::integral_constant<int, 1>());
        } else {
            if (p.rs_chains >= 4) walk0s(uint32_t(), std::integral_constant<int, 4>());
            else if (p.rs_chains == 2) walk0s(uint32_t(), std::integral_constant<int, 2>());
            else walk0s(uint32_t(), std::integral_constant<int, 1>());
        }
        phase_end(c, s, PH_WALK0);
    } else if (L.direct && !U) {
        phase_begin(c, s);
        rs_walk_direct<<<(unsigned)((L0.nb + BLOCK - 1) / BLOCK), BLOCK, 0, s>>>(
            succ, reinterpret_cast<uint32_t*>(rank), L0, L.pbits, (int)(L.size[1] - L.fixed), R(1), ctl);
        phase_end(c, s, PH_WALK0);
    } else if (L.values) {
        phase_begin(c, s);
        rs_walk_values<true><<<(unsigned)((L0.nb + BLOCK - 1) / BLOCK), BLOCK, 0, s>>>(
            W0, reinterpret_cast<uint64_t*>(base + L.off_P0), L0, R(1), ctl);
        phase_end(c, s, PH_WALK0);
    } else if (!U) {
        walk0();
    }
    for (int l = 1; l < L.levels; ++l) {
        const uint32_t seed = mix32(seed0 + 0x9E3779B9u * (uint32_t)l);
        const unsigned g = (unsigned)((L.size[l + 1] + BLOCK - 1) / BLOCK);
        phase_begin(c, s);
        const uint32_t fixed = l == 1 && L.fixed > 0 ? (uint32_t)L.fixed : 0xFFFFFFFFu;
        if (val)
            rs_chase<true><<<g, BLOCK, 0, s>>>(R(l), (uint32_t)L.size[l], P(l), R(l + 1), (uint32_t)L.size[l + 1],
                                               L.logD[l], seed, fixed, &ctl->chased[l], ctl);
        else
            rs_chase<false><<<g, BLOCK, 0, s>>>(R(l), (uint32_t)L.size[l], P(l), R(l + 1), (uint32_t)L.size[l + 1],
                                                L.logD[l], seed, fixed, nullptr, ctl);
        phase_end(c, s, PH_WALK);
    }
    {
        const int lf = L.levels;
        const int r = (int)L.size[lf];
        const size_t smem = br_smem(r);
        phase_begin(c, s);
        allow_smem(c, (const void*)rs_final_kernel, br_smem(16384));
        rs_final_kernel<<<1, FINAL_THREADS, smem, s>>>(R(lf), r, lf == 1 && L.fixed > 0 ? (int)L.fixed : r, S(lf),
                                                       val ? -1 : n, L.values ? (unsigned long long)n : 0ull,
                                                       U ? U->head_dev + 5 : nullptr, seed0, ctl);
        phase_end(c, s, PH_FINAL);
    }
    for (int l = L.levels - 1; l >= 1; --l) {
        const int g = stream_grid(c, L.size[l], (const void*)rs_expand);
        phase_begin(c, s);
        rs_expand<<<g, BLOCK, 0, s>>>(P(l), (uint32_t)L.size[l], S(l + 1), (uint32_t)L.size[l + 1], S(l),
                                     val ? &ctl->chased[l] : nullptr, ctl);
        phase_end(c, s, PH_EXPAND);
    }
    if (L.readonly) {
        phase_begin(c, s);
        allow_smem(c, (const void*)rs_scatter, SC_SMEM);
        const int gs = std::min((int)L.grid, persistent_grid(c, (const void*)rs_scatter, BLOCK, SC_SMEM));
        rs_scatter<<<gs, BLOCK, SC_SMEM, s>>>(C, (int)L.grid, S(1), W0, n, ctl);
        phase_end(c, s, PH_SCATTER);
        phase_begin(c, s);
        rs_place<<<LRCC_PLACE_BLOCKS_PER_SM * c->sms, BLOCK, 0, s>>>(W0, n, rank, ctl);
        phase_end(c, s, PH_EXPAND0);
    } else if (L.split) {
        phase_begin(c, s);
        if (mark16) {
            const int g = stream_grid(c, n, (const void*)rs_expand0s<uint16_t>);
            rs_expand0s<uint16_t><<<g, BLOCK, 0, s>>>((const uint16_t*)mark, lrank, n, S(1), L.size[1], rank, ctl);
        } else {
            const int g = stream_grid(c, n, (const void*)rs_expand0s<uint32_t>);
            rs_expand0s<uint32_t><<<g, BLOCK, 0, s>>>((const uint32_t*)mark, lrank, n, S(1), L.size[1], rank, ctl);
        }
        phase_end(c, s, PH_EXPAND0);
    } else if (L.direct && U) {
        // (below)
    } else if (L.direct) {
        const bool v = aligned16(rank);
        const void* k = v ? (const void*)rs_expand_direct<true> : (const void*)rs_expand_direct<false>;
        const int g = stream_grid(c, groups, k);
        phase_begin(c, s);
        if (v) rs_expand_direct<true><<<g, BLOCK, 0, s>>>(rank, n, S(1), (uint32_t)L.size[1], L.pbits);
        else rs_expand_direct<false><<<g, BLOCK, 0, s>>>(rank, n, S(1), (uint32_t)L.size[1], L.pbits);
        phase_end(c, s, PH_EXPAND0);
    } else if (L.values) {
        const uint32_t* S1 = reinterpret_cast<const uint32_t*>(S(1));
        enqueue_expand_values(c, s, reinterpret_cast<uint64_t*>(base + L.off_P0), n, S1, 1, 0, L.size[1], rank);
    } else {
        const bool v = vec && aligned16(rank);
        const void* k = v ? (const void*)rs_expand0<true> : (const void*)rs_expand0<false>;
        const int g = stream_grid(c, groups, k);
        phase_begin(c, s);
        const int bias = val ? 0 : 1;
        if (v) rs_expand0<true><<<g, BLOCK, 0, s>>>(W0, n, S(1), L.size[1], rank, bias, ctl);
        else rs_expand0<false><<<g, BLOCK, 0, s>>>(W0, n, S(1), L.size[1], rank, bias, ctl);
        phase_end(c, s, PH_EXPAND0);
    }
    if (L.direct && U) {
        auto expand = [&](auto v, auto again) {
            auto k = rs_expand_lists<decltype(v)::value, decltype(again)::value>;
            phase_begin(c, s);
            k<<<stream_grid(c, groups, (const void*)k), BLOCK, 0, s>>>(rank, n, S(1), (uint32_t)L.size[1], L.pbits, U->off,
                                                                       U->K, U->head_dev, succ, U->heads,
                                                                       static_cast<uint64_t*>(c->ws), seed0, ctl);
            phase_end(c, s, PH_EXPAND0);
        };
        if (aligned16(rank))
            U->again ? expand(std::true_type(), std::true_type()) : expand(std::true_type(), std::false_type());
        else
            U->again ? expand(std::false_type(), std::true_type()) : expand(std::false_type(), std::false_type());
    }
    return cuda_status(cudaGetLastError());
}

// Forest layout: walk words W0 (8 B per element), the has-predecessor bitmap, the
// elements' records (8 B, up to WALK_NEAR elements: above they are kept in W0), and for
// r1_max = nb + n first-level splitters (every element could be a head) their packed
// words and the extra ones' elements (12 B): 21 bytes per element, 30 up to WALK_NEAR.
struct ForestLayout {
    int logD;
    int64_t nb, r1_max;
    size_t off_W0, off_pred, off_P0, off_R1, off_extra, bytes;
};

ForestLayout forest_layout(int64_t n, int spacing0) {
    ForestLayout F;
    F.logD = 2;
    while (F.logD < 20 && (int64_t(1) << (F.logD + 1)) <= spacing0) ++F.logD;
    F.nb = (n + (int64_t(1) << F.logD) - 1) >> F.logD;
    F.r1_max = F.nb + n;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off = align_up(off + bytes, 256);
        return o;
    };
    F.off_W0 = take(sizeof(uint64_t) * (size_t)n);
    F.off_pred = take(sizeof(uint32_t) * (size_t)((n + 31) / 32));
    F.off_P0 = n <= WALK_NEAR ? take(sizeof(uint64_t) * (size_t)n) : F.off_W0;
    F.off_R1 = take(sizeof(uint64_t) * (size_t)F.r1_max);
    F.off_extra = take(sizeof(int32_t) * (size_t)F.r1_max);
    F.bytes = off;
    return F;
}

size_t lr_scan_forest_ws(int64_t n, const Plan& p) { return forest_layout(n, p.rs_spacing0).bytes; }

lrcc_status lr_enqueue_scan_forest(Ctx* c, cudaStream_t s, const int32_t* succ, const int32_t* val, int64_t n,
                                   int32_t* out, const Plan& p) {
    const ForestLayout F = forest_layout(n, p.rs_spacing0);
    char* base = static_cast<char*>(c->ws);
    uint64_t* W0 = reinterpret_cast<uint64_t*>(base + F.off_W0);
    uint32_t* pred = reinterpret_cast<uint32_t*>(base + F.off_pred);
    uint64_t* P0 = reinterpret_cast<uint64_t*>(base + F.off_P0);
    uint64_t* R1 = reinterpret_cast<uint64_t*>(base + F.off_R1);
    int32_t* extra = reinterpret_cast<int32_t*>(base + F.off_extra);
    DevCtl* ctl = c->ctl;
    Level0 L0;
    L0.n = n;
    L0.nb = F.nb;
    L0.logD = F.logD;
    L0.seed = (uint32_t)(p.seed ^ (p.seed >> 32));
    // no head among the stratified splitters: block 0 keeps its own
    L0.bh = 0;
    L0.head_off = (uint32_t)((uint64_t)mix32(L0.seed) * (uint64_t)std::min<int64_t>(n, int64_t(1) << F.logD) >> 32);
    L0.extra = extra;
    L0.extra_count = &ctl->ff_extra;
    cudaMemsetAsync(pred, 0, sizeof(uint32_t) * (size_t)((n + 31) / 32), s);
    phase_begin(c, s);
    ff_links<<<stream_grid(c, (n + 3) / 4, (const void*)ff_links), BLOCK, 0, s>>>(succ, n, pred, ctl);
    ff_select<<<stream_grid(c, (n + 3) / 4, (const void*)ff_select), BLOCK, 0, s>>>(succ, val, n, pred, W0, extra, L0, ctl);
    phase_end(c, s, PH_SELECT0);
    phase_begin(c, s);
    // (a few heads more than nb threads are left to the stride)
    const unsigned gw = (unsigned)((F.nb + BLOCK - 1) / BLOCK);
    if (P0 != W0) rs_walk_values<true><<<gw, BLOCK, 0, s>>>(W0, P0, L0, R1, ctl);
    else rs_walk_values<false><<<gw, BLOCK, 0, s>>>(W0, P0, L0, R1, ctl);
    phase_end(c, s, PH_WALK0);
    phase_begin(c, s);
    {
        GangCtl* gc = reinterpret_cast<GangCtl*>(reinterpret_cast<char*>(ctl) + offsetof(DevCtl, gang));
        int64_t nn = n, nb = F.nb;
        uint64_t* words = R1;
        void* args[] = {&words, &nn, &nb, &gc, &ctl};
        const int blocks = (int)std::min<int64_t>(c->sms, (F.nb + GANG_THREADS - 1) / GANG_THREADS);
        if (cudaLaunchCooperativeKernel((const void*)ff_rounds, dim3(blocks), dim3(GANG_THREADS), args, 0, s) != cudaSuccess)
            return LRCC_ERR_CUDA;
    }
    phase_end(c, s, PH_WY_JUMP);
    enqueue_expand_values(c, s, P0, n, reinterpret_cast<uint32_t*>(R1), 2, 1, F.r1_max, out);
    return cuda_status(cudaGetLastError());
}

lrcc_status lr_enqueue_wyllie(Ctx* c, cudaStream_t s, const int32_t* succ, int64_t n, int32_t head,
                              int32_t* rank, const Plan& p) {
    if (n <= p.rs_small) return launch_small_wyllie(c, s, succ, (int)n, head, rank);
    uint64_t* W0 = static_cast<uint64_t*>(c->ws);
    uint64_t* W1 = reinterpret_cast<uint64_t*>(static_cast<char*>(c->ws) +
                                               align_up(sizeof(uint64_t) * (size_t)n, 256));
    const int64_t groups = (n + 3) / 4;
    const bool vec = aligned16(succ) && aligned16(rank);
    {
        const void* k = vec ? (const void*)wy_pack<true> : (const void*)wy_pack<false>;
        const int g = stream_grid(c, groups, k);
        phase_begin(c, s);
        if (vec) wy_pack<true><<<g, BLOCK, 0, s>>>(succ, n, W0, c->ctl);
        else wy_pack<false><<<g, BLOCK, 0, s>>>(succ, n, W0, c->ctl);
        phase_end(c, s, PH_WY_PACK);
    }
    int rounds = 0;
    while ((int64_t(1) << rounds) < n) ++rounds;
    const int gj = stream_grid(c, groups, (const void*)wy_jump);
    uint64_t* a = W0;
    uint64_t* b = W1;
    for (int r = 0; r + 1 < rounds; ++r) {
        phase_begin(c, s);
        wy_jump<<<gj, BLOCK, 0, s>>>(a, b, n);
        phase_end(c, s, PH_WY_JUMP);
        std::swap(a, b);
    }
    {
        const void* k = vec ? (const void*)wy_final<true> : (const void*)wy_final<false>;
        const int g = stream_grid(c, groups, k);
        phase_begin(c, s);
        if (vec) wy_final<true><<<g, BLOCK, 0, s>>>(a, n, head, rank, c->ctl);
        else wy_final<false><<<g, BLOCK, 0, s>>>(a, n, head, rank, c->ctl);
        phase_end(c, s, PH_WY_FINAL);
    }
    return cuda_status(cudaGetLastError());
}

}  // namespace lrcc
