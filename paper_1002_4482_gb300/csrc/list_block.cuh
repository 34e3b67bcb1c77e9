// One list of a batch ranked by one thread block in global memory, by the kernels
// that rank lists one by one (batch.cu) and, when ranking them together failed, by
// the one that would have expanded their ranks (lr.cu).
#pragma once

#include "block_rank.cuh"
#include "common.cuh"

namespace lrcc {

__device__ __forceinline__ int64_t take_instance(int* s_k, int* next, int64_t count) {
    __syncthreads();
    if (threadIdx.x == 0) *s_k = atomicAdd(next, 1);
    __syncthreads();
    return *s_k < count ? *s_k : -1;
}

// Whether a list of n elements from element b on lies in a call's `total` elements.
__device__ __forceinline__ bool list_in_range(int64_t b, int64_t n, int64_t total) {
    return b >= 0 && n >= 0 && b <= total && n <= total - b;
}

// Rank one larger list with a ruling set inside the block; W is the list's
// slice of the 8-byte word workspace, R the splitters' packed words in shared
// memory (next splitter, sublist length; before the walk: successor, 1). Indices
// read back from W are checked: offsets that overlap (reported) put two blocks on
// the same words.
template <int T, int CAP>
__device__ void list_ruling_set(const int32_t* succ, int64_t n, int head, int32_t* rank, uint64_t* W,
                                uint64_t* R, uint2* sub, int* s_work, uint32_t seed, int min_logD, DevCtl* ctl) {
    // spacing: a power of two, at least 2^min_logD, with at most CAP splitters
    int logD = max(2, min_logD);
    while (((n + (int64_t(1) << logD) - 1) >> logD) > CAP) ++logD;
    const int64_t D = int64_t(1) << logD;
    const int r = (int)((n + D - 1) >> logD);
    const int64_t bh = head >> logD;
    const uint32_t head_off = (uint32_t)(head - (bh << logD));
    // select (RS1+RS2): walk words, and each splitter's successor in R[j]
    for (int64_t i = threadIdx.x; i < n; i += T) {
        const int s = succ[i];
        const bool tail = (s == -1) | (s == i);
        const bool bad = !tail && (s < 0 || s >= n);
        if (bad) record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)i);
        const uint32_t nx = (tail || bad) ? NIL : (uint32_t)s;
        const int64_t b = i >> logD;
        const uint32_t size = (uint32_t)min(D, n - (b << logD));
        const uint32_t off = b == bh ? head_off : block_offset((uint32_t)b, size, seed);
        if ((uint32_t)(i - (b << logD)) == off) {
            const int j = (int)(b >= bh ? b - bh : b - bh + r);
            W[i] = pack(nx | SPL, (uint32_t)j);
            R[j] = pack(nx, 1);
        } else {
            W[i] = pack(nx, 1);
        }
    }
    if (threadIdx.x == 0) *s_work = 0;
    __syncthreads();
    // walk (RS3): one sublist per thread at a time, claimed from a shared counter
    for (;;) {
        const int j = atomicAdd(s_work, 1);
        if (j >= r) break;
        uint32_t cur = lo32(R[j]);
        uint32_t pre = 1;
        uint32_t next = NIL;
        int64_t steps = 0;
        while (cur != NIL) {
            if (cur >= n) {
                record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)cur);
                break;
            }
            const uint64_t w = W[cur];
            const uint32_t lo = lo32(w), hi = hi32(w);
            if (lo & SPL) {
                if (hi < (uint32_t)r) next = hi;
                break;
            }
            if ((hi & VIS) || ++steps > n) {
                record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)cur);
                break;
            }
            W[cur] = pack(pre, (uint32_t)j | VIS);
            pre += hi;
            cur = lo;
        }
        R[j] = pack(next == NIL ? BR_NIL : next, pre);
    }
    // rank the splitters (RS4) in shared memory; their suffix sums replace their words
    bool whole;
    const uint2* res = block_rank<T>(R, sub, r, 0, seed, &whole, ctl);
    if (threadIdx.x == 0 && (!whole || (int64_t)res[0].y != n)) record_error(ctl, LRCC_ERR_INVALID_INPUT, -3);
    for (int j = threadIdx.x; j < r; j += T) R[j] = (uint64_t)(uint32_t)block_rank_sum<T>(R[j], res);
    __syncthreads();
    // expand (RS5)
    for (int64_t i = threadIdx.x; i < n; i += T) {
        const uint64_t w = W[i];
        const uint32_t lo = lo32(w), hi = hi32(w);
        int out;
        if ((lo & SPL) && hi < (uint32_t)r) {
            out = (int)lo32(R[hi]) - 1;
        } else if (!(lo & SPL) && (hi & VIS) && (hi & ~VIS) < (uint32_t)r) {
            out = (int)lo32(R[hi & ~VIS]) - (int)lo - 1;
        } else {
            record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)i);
            out = -1;
        }
        rank[i] = out;
    }
}

}  // namespace lrcc
