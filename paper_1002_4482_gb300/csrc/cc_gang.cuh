// Building blocks of the component kernels that keep a whole graph's rounds in
// one launch: a gang of blocks with its own barrier, edge passes over
// warp-private ranges, and active edges kept as pairs of roots.
#pragma once

#include "cc_device.cuh"
#include "common.cuh"

namespace lrcc {

constexpr int GANG_THREADS = 1024;
constexpr int GANG_WARPS = GANG_THREADS / 32;
constexpr int GANG_EDGES = 4;                 // edges per lane and iteration
constexpr int GANG_STEP = 32 * GANG_EDGES;    // edges per warp and iteration

// Shared state of one gang in device memory, zero before the launch.
struct GangCtl {
    unsigned arrived[2];     // barrier arrivals so far, one counter per launch
    unsigned pad0[30];
    unsigned long long kept[3];   // edges kept by the pass (three passes in rotation)
    unsigned pad1[26];
};

// A barrier over the gang's blocks, all of them resident (cooperative launch).
// Everything written before it by any block is visible after it. The wait is
// bounded: after about two seconds it records LRCC_ERR_TIMEOUT and returns
// false, and the kernel returns. 1.2-1.5 us for 152 blocks, against 8.3 us for
// one iteration of a while-node with three kernels.
struct Gang {
    GangCtl* g;
    unsigned* arrived;       // this launch's counter
    int size, rank;          // blocks of the gang, this block's place
    unsigned target;         // arrivals that complete the next barrier
    DevCtl* ctl;
    int* s_flag;             // shared memory

    __device__ __forceinline__ bool sync() {
        __syncthreads();
        if (size > 1) {
            if (threadIdx.x == 0) {
                target += (unsigned)size;
                asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(arrived) : "memory");
                bool ok = false;
                for (int i = 0; i < (1 << 23) && !ok; ++i) {
                    unsigned v;
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(arrived) : "memory");
                    ok = (int)(v - target) >= 0;
                }
                if (!ok) record_error(ctl, LRCC_ERR_TIMEOUT, -8);
                *s_flag = ok;
            }
            __syncthreads();
            return *s_flag != 0;
        }
        return true;
    }
    __device__ __forceinline__ int warps() const { return size * GANG_WARPS; }
    __device__ __forceinline__ int warp() const { return rank * GANG_WARPS + (int)(threadIdx.x >> 5); }
};

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
// 1 G/s. So the lanes that hook the same root send one atomic with the smallest
// of their ids, and a block remembers the roots it hooks: slot -> (root,
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

}  // namespace lrcc
