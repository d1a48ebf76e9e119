// kg_resident.cuh -- arguments, launch and counting-sort phases shared by the three
// resident MD kernels (kg_resident.cu, kg_resident_small.cu, kg_resident_tiled.cu).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>

#include "kg_gridbar.cuh"
#include "kg_step.cuh"

namespace kg {

constexpr int RES_SEG = 1024;            // cells per scan segment

struct ResArgs {
    StepArgs st;                 // its dcur/dnext/pcur/pnext are ignored: the buffers alternate below
    NlArgs nl;
    const SimDev *sim;           // device copy of the melt table (binning)
    float4 *dlt[2], *pg[2];      // displacement and gather buffers, ping-pong
    double *x, *xb64;
    float4 *recb, *recs;
    int *cellid, *rank, *ccount, *cstart, *clist, *ctmp, *segtot;
    int *count[2], *bidx;        // small kernel: bucket counts (the set named by flags[RES_NEXT] is zero between
    float4 *brec, *brec2;        //   rebuilds), members in arrival order, records in order (w = compute index)
    int ncell, cur0, K, skip_block;   // skip_block >= 0: that block never arrives (barrier self-test)
    unsigned long long *bar;     // three barrier words, zero at launch
    unsigned *errw;              // error bits of this launch (zero at launch)
    unsigned spin;               // barrier polls before giving up
    long long *stepp;            // device step counter: the last step run
};

// total of segment g of the cell counts (block of NT threads; wsum: NT / 32 words)
template <int NT>
__device__ __forceinline__ void res_seg_total(const ResArgs &A, const int *count, int g, int *wsum)
{
    int t = 0;
    for (int k = threadIdx.x; k < RES_SEG; k += NT) t += g * RES_SEG + k < A.ncell ? count[g * RES_SEG + k] : 0;
    t = __reduce_add_sync(0xffffffffu, t);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < NT / 32; ++w) t += wsum[w];
        A.segtot[g] = t;
    }
    __syncthreads();
}

// exclusive scan of the cell counts: segment g from the totals of the segments
// before it and its own counts (wsum: NT / 16 words)
template <int NT>
__device__ __forceinline__ void res_scan_seg(const ResArgs &A, const int *count, int g, int nseg, int *wsum)
{
    constexpr int PER = RES_SEG / NT, NW = NT / 32;
    const int n = A.ncell, i0 = g * RES_SEG + threadIdx.x * PER;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int before = 0;
    for (int k = threadIdx.x; k < g; k += NT) before += A.segtot[k];
    int v[PER], own = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        v[k] = i0 + k < n ? count[i0 + k] : 0;
        own += v[k];
    }
    int incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    before = __reduce_add_sync(0xffffffffu, before);
    if (lane == 31) wsum[w] = incl;
    if (lane == 0) wsum[NW + w] = before;
    __syncthreads();
    int run = incl - own;
#pragma unroll
    for (int k = 0; k < NW; ++k) run += wsum[NW + k] + (k < w ? wsum[k] : 0);
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        if (i0 + k < n) A.cstart[i0 + k] = run;
        run += v[k];
    }
    if (g == nseg - 1 && threadIdx.x == NT - 1) A.cstart[n] = run;
    __syncthreads();
}

// launches kernel K<N4> of the context's stage exponent on `blocks` cooperative blocks
#define KG_RESIDENT_LAUNCH(K, n4, blocks, threads, a, st)                                                             \
    [&]() -> cudaError_t {                                                                                             \
        cudaLaunchConfig_t cfg{};                                                                                      \
        cfg.gridDim = dim3((unsigned)(blocks));                                                                        \
        cfg.blockDim = dim3(threads);                                                                                  \
        cfg.stream = st;                                                                                               \
        cudaLaunchAttribute attr[1];                                                                                   \
        attr[0].id = cudaLaunchAttributeCooperative;                                                                   \
        attr[0].val.cooperative = 1;                                                                                   \
        cfg.attrs = attr;                                                                                              \
        cfg.numAttrs = 1;                                                                                              \
        switch (n4) {                                                                                                  \
            case 8: return cudaLaunchKernelEx(&cfg, K<8>, a);                                                          \
            case 12: return cudaLaunchKernelEx(&cfg, K<12>, a);                                                        \
            case 16: return cudaLaunchKernelEx(&cfg, K<16>, a);                                                        \
            case 20: return cudaLaunchKernelEx(&cfg, K<20>, a);                                                        \
            case 23: return cudaLaunchKernelEx(&cfg, K<23>, a);                                                        \
            case 26: return cudaLaunchKernelEx(&cfg, K<26>, a);                                                        \
            case 28: return cudaLaunchKernelEx(&cfg, K<28>, a);                                                        \
            case 32: return cudaLaunchKernelEx(&cfg, K<32>, a);                                                        \
            case 36: return cudaLaunchKernelEx(&cfg, K<36>, a);                                                        \
            case 40: return cudaLaunchKernelEx(&cfg, K<40>, a);                                                        \
            case 44: return cudaLaunchKernelEx(&cfg, K<44>, a);                                                        \
            case 48: return cudaLaunchKernelEx(&cfg, K<48>, a);                                                        \
            default: return cudaLaunchKernelEx(&cfg, K<0>, a);                                                         \
        }                                                                                                              \
    }()

// kg_resident_small.cu
constexpr int SMALL_OWN = 64, SMALL_MIN_BLOCKS = 2;   // monomers of a block of the small kernel, blocks per SM
cudaError_t small_launch(const ResArgs &a, int n4, cudaStream_t st);
// kg_resident_tiled.cu
cudaError_t tiled_launch(const ResArgs &a, int n4, int sms, cudaStream_t st);

}  // namespace kg
