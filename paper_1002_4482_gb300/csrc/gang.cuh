// A gang: blocks of one cooperative launch that work together behind a barrier of
// their own (a whole grid, or one of several gangs in it).
#pragma once

#include "common.cuh"

namespace lrcc {

constexpr int GANG_THREADS = 1024;
constexpr int GANG_WARPS = GANG_THREADS / 32;

// Shared state of one gang in device memory, zero before the launch.
struct GangCtl {
    unsigned arrived[2];     // barrier arrivals so far, one counter per launch
    unsigned instance;       // batched: the instance the gang works on
    unsigned pad0[29];
    unsigned long long kept[3];   // edges kept by the pass (three passes in rotation)
    unsigned pad1[26];
};

// A barrier over the gang's blocks, all of them resident (cooperative launch).
// Everything written before it by any block is visible after it. The wait is
// bounded: after about two seconds it records LRCC_ERR_TIMEOUT, marks the call
// (DevCtl::gave_up, for launches that follow) and returns false, and the kernel
// returns. 1.2-1.5 us for 152 blocks, against 8.3 us for
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
                if (!ok) {
                    record_error(ctl, LRCC_ERR_TIMEOUT, -8);
                    ctl->gave_up = 1;
                }
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

}  // namespace lrcc
