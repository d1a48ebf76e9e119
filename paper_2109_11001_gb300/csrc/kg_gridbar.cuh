// kg_gridbar.cuh -- grid barrier of the cooperative kernels (resident MD loop,
// double-bridging commit rounds), with bounded waits.
#pragma once
#include <cuda_runtime.h>

namespace kg {

// fields of a barrier word: blocks arrived, blocks asking for a rebuild, that saw an error, with a full bucket
constexpr unsigned long long BAR_MASK = 0xffffull;
constexpr unsigned REQ = 1u, FAIL = 2u, OVER = 4u, GAVE_UP = 8u;      // what a barrier tells

struct GridBar {
    unsigned long long *bar;
    unsigned *acc, *out;         // shared: this block's bits for the next barrier [2], the last barrier's answer
    unsigned spin;
    int b;                       // barriers passed

    // bits of any thread reach the barrier that the block arrives at next
    __device__ __forceinline__ void note(unsigned bits) { if (bits) atomicOr(acc + (b & 1), bits); }

    // every thread's stores and notes go first
    __device__ __forceinline__ void arrive()
    {
        __syncthreads();
        arrive_as_is();
    }

    __device__ __forceinline__ void arrive_as_is()
    {
        if (threadIdx.x == 0) {
            const unsigned a = acc[b & 1];
            acc[(b + 1) & 1] = 0u;
            if (blockIdx.x == 0) *(volatile unsigned long long *)(bar + (b + 1) % 3) = 0ull;
            const unsigned long long add = 1ull + ((unsigned long long)(a & REQ) << 16) +
                                           ((unsigned long long)((a & FAIL) >> 1) << 32) +
                                           ((unsigned long long)((a & OVER) >> 2) << 48);
            // the fence orders the whole block's stores (the block barrier before it) before the arrival
            asm volatile("fence.acq_rel.gpu;\n\tred.relaxed.gpu.global.add.u64 [%0], %1;"
                         ::"l"(bar + b % 3), "l"(add) : "memory");
        }
    }

    __device__ __forceinline__ unsigned wait()
    {
        if (threadIdx.x == 0) {
            unsigned long long v;
            unsigned it = 0, r = 0;
            for (;;) {
                asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(bar + b % 3) : "memory");
                if ((v & BAR_MASK) == gridDim.x) break;
                if (++it > spin) {
                    r = GAVE_UP;
                    break;
                }
                if (it > 64) __nanosleep(32);
            }
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
            if ((v >> 16) & BAR_MASK) r |= REQ;
            if ((v >> 32) & BAR_MASK) r |= FAIL;
            if (v >> 48) r |= OVER;
            *out = r;
        }
        __syncthreads();
        ++b;
        return *out;
    }

    __device__ __forceinline__ unsigned sync()
    {
        arrive();
        return wait();
    }
};

}  // namespace kg
