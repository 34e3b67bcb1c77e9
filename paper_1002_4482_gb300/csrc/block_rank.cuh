// Ranking of a linked list held in shared memory by one thread block: a sparse
// ruling set (Sec. 3.2) whose splitters, one per thread, are ranked by pointer
// jumping (Sec. 3.1, the single-block variant). It ranks the last level of the
// recursive ruling set and every list that fits one block.
//
// Pointer jumping over all r elements does r log2 r shared-memory gathers of
// two words, 14 rounds of 16 elements per thread at r = 16384; here every
// element is read and written once by the walk and once by the expansion, and
// only the splitters jump. The walk is bound by the latency of its longest
// sublist (about D ln(THREADS) dependent shared-memory reads of some 30 cycles
// each), so the spacing D is the smallest power of two that leaves one
// splitter per thread. A list of 100,003 elements, whose last level has 12,501
// splitters, is ranked in 66.6 us against 98.3 with pointer jumping over them
// all; one of 2^20 (8192 splitters) in 138.6 against 155.3.
#pragma once

#include "common.cuh"

namespace lrcc {

// Packed words in shared memory: low half = next element or BR_NIL, high half
// = weight; the walk overwrites a word with (owner | flag, prefix weight).
constexpr uint32_t BR_NIL = 0x3FFFFFFFu;
constexpr uint32_t BR_VIS = 0x40000000u;   // visited by a walk
constexpr uint32_t BR_SPL = 0x80000000u;   // a splitter (prefix weight 0)
constexpr uint32_t BR_OWNER = 0x3FFFFFFFu;
constexpr uint32_t BR_END = 0xFFFu;        // splitter words: no next splitter
constexpr int BR_CNT = 12;                 // splitter words: next in the low 12 bits, element count above

// W[0..r) holds one list with the given head (r < 2^20, THREADS < 4095), sub is
// scratch for 2 * THREADS words. Returns the splitters' words: for element i,
// owner o = lo32(W[i]) & BR_OWNER, the weights from i to the tail (inclusive,
// modulo 2^32) sum to result[o].y - hi32(W[i]). *whole is set to whether the
// elements form one list from head that holds all r of them; a cycle, or an
// element reached twice, is recorded as invalid input as well. All threads
// call it; the words may be read when it returns.
template <int THREADS>
__device__ const uint2* block_rank(uint64_t* W, uint2* sub, int r, int head, uint32_t seed, bool* whole,
                                   DevCtl* ctl) {
    static_assert(THREADS < (int)BR_END, "splitter indices fit their field");
    const int t = threadIdx.x;
    int logD = 0;
    while (((r + (1 << logD) - 1) >> logD) > THREADS) ++logD;
    const int nsub = (r + (1 << logD) - 1) >> logD;
    uint32_t cur = BR_NIL, pre = 0, cnt = 0;
    __syncthreads();   // the words are loaded
    if (t < nsub) {
        // one splitter per block of 2^logD elements at a hashed offset; the
        // head's block takes the head
        const int base = t << logD;
        const int off = t == (head >> logD) ? head - base : (int)block_offset(t, min(1 << logD, r - base), seed);
        const uint64_t w = W[base + off];
        cur = lo32(w);
        pre = hi32(w);
        cnt = 1;
        W[base + off] = pack((uint32_t)t | BR_SPL, 0);
    }
    __syncthreads();
    uint32_t next = BR_END;
    while (cur != BR_NIL) {
        const uint64_t w = W[cur];
        const uint32_t lo = lo32(w);
        if (lo & BR_SPL) {
            next = lo & BR_OWNER;
            break;
        }
        if (lo & BR_VIS) {   // reached twice: not a list
            record_error(ctl, LRCC_ERR_INVALID_INPUT, (int)cur);
            break;
        }
        W[cur] = pack((uint32_t)t | BR_VIS, pre);
        pre += hi32(w);
        ++cnt;
        cur = lo;
    }
    // pointer jumping over the splitters, one per thread, between two buffers
    int at = 0;
    sub[t] = make_uint2(next | (cnt << BR_CNT), pre);
    int cap = 2;
    while ((1 << (cap - 2)) < nsub) ++cap;
    __syncthreads();
    for (int round = 0;; ++round) {
        if (next != BR_END) {
            const uint2 o = sub[at * THREADS + next];
            next = o.x & BR_END;
            cnt += o.x >> BR_CNT;
            pre += o.y;
        }
        at ^= 1;
        sub[at * THREADS + t] = make_uint2(next | (cnt << BR_CNT), pre);
        if (!__syncthreads_or(next != BR_END)) break;
        if (round >= cap) {   // links left after ceil(log2) rounds: a cycle
            if (t == 0) record_error(ctl, LRCC_ERR_INVALID_INPUT, -2);
            break;
        }
    }
    const uint2* res = sub + at * THREADS;
    *whole = (res[head >> logD].x >> BR_CNT) == (uint32_t)r;
    return res;
}

// Weights from element i to the tail, inclusive. A word that no walk reached
// (possible only after an error) gives an owner outside the block: 0 then.
template <int THREADS>
__device__ __forceinline__ int block_rank_sum(uint64_t w, const uint2* res) {
    const uint32_t o = lo32(w) & BR_OWNER;
    return (lo32(w) & (BR_SPL | BR_VIS)) && o < (uint32_t)THREADS ? (int)(res[o].y - hi32(w)) : 0;
}

}  // namespace lrcc
