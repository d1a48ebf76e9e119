// kg_resident.cu -- the mixed path's MD loop for systems whose monomers all fit
// the GPU's resident threads: one cooperative launch runs K steps, one thread
// per monomer.
//
// What bounds a small system is not work but the chain of dependent waits: as
// separate launches a step is a begin kernel, a conditional graph node and a
// step kernel, each a launch of several microseconds around one or two
// microseconds of load latency.  Here a step is one grid barrier and one round
// of gathers:
//  * a thread keeps its monomer's velocity, displacement, build record, list
//    length, chain partners and slot in registers from step to step; per step
//    it loads its list entries and the gather records of its neighbours and
//    partners and stores its own gather record;
//  * STEP_ILP list entries and their gathers are in flight together (8 here, 4
//    in the one-step kernel, whose latency is hidden by resident warps instead);
//  * the barrier is split: a block arrives as soon as its gather records are
//    stored, draws the noise of the next step, and then waits;
//  * the barrier word itself counts the blocks that ask for a list rebuild or
//    saw an error, so a waiting block learns both with the poll that releases
//    it.  Three words rotate: word b % 3 serves barrier b, and block 0 clears
//    word (b + 1) % 3 before it arrives at barrier b (its last readers left
//    at barrier b - 2).
// The Verlet rebuild runs between barriers of the same kind: bin (which also
// totals the counts of every 1024-cell segment), scan of the cell counts,
// scatter, in-cell rank, list.
//
// Every wait is bounded by a poll count, after which the block latches
// ERR_TIMEOUT and leaves.  The arithmetic is that of the one-step kernel
// (kg_step.cuh) on the same lists, so trajectories have the same bits.
//
// Measured, 50 steps and the read of the state (skin 0.3, n = 12, dt = 0.01; a
// build every third or fourth step), against the captured graphs of separate
// launches: 1,000 monomers 1230 -> 613 us, 16 melts of 1,000 in one context
// 1998 -> 1362 us (about half of it the reads), 80,000 monomers 1674 -> 1170 us.
// Larger systems keep the graphs: there the step is work and the launches are
// not.
//
// (128, 5): at most 102 registers, 5 x 128 threads per SM; the capacity (about
// 97,000 monomers on 152 SMs) is resident_fits' limit.
#include <cuda_runtime.h>

#include <algorithm>

#include "kg_step.cuh"

namespace kg {

constexpr int RES_BLOCK = 128;
constexpr int RES_MIN_BLOCKS = 5;
constexpr int RES_ILP = 8;               // list entries in flight per lane
constexpr int RES_SEG = 1024;            // cells per scan segment

struct ResArgs {
    StepArgs st;                 // its dcur/dnext/pcur/pnext are ignored: the buffers alternate below
    NlArgs nl;
    const SimDev *sim;           // device copy of the melt table (binning)
    float4 *dlt[2], *pg[2];      // displacement and gather buffers, ping-pong
    double *x, *xb64;
    float4 *recb, *recs;
    int *cellid, *rank, *ccount, *cstart, *clist, *ctmp, *segtot;
    int ncell, cur0, K, skip_block;   // skip_block >= 0: that block never arrives (barrier self-test)
    unsigned long long *bar;     // three barrier words, zero at launch
    unsigned *errw;              // error bits of this launch (zero at launch)
    unsigned spin;               // barrier polls before giving up
    long long *stepp;            // device step counter: the last step run
};

// fields of a barrier word: blocks arrived, blocks asking for a rebuild, blocks that saw an error
constexpr unsigned long long BAR_ONE = 1ull, BAR_REQ = 1ull << 21, BAR_ERR = 1ull << 42;
constexpr unsigned long long BAR_MASK = (1ull << 21) - 1ull;
constexpr unsigned REQ = 1u, FAIL = 2u, GAVE_UP = 4u;       // what a barrier tells

struct GridBar {
    unsigned long long *bar;
    unsigned *acc, *out;         // shared: this block's bits for the next barrier [2], the last barrier's answer
    unsigned spin;
    int b;                       // barriers passed

    // bits of any thread reach the barrier that the block arrives at next
    __device__ __forceinline__ void note(unsigned bits) { if (bits) atomicOr(acc + (b & 1), bits); }

    __device__ __forceinline__ void arrive()
    {
        __syncthreads();
        if (threadIdx.x == 0) {
            const unsigned a = acc[b & 1];
            acc[(b + 1) & 1] = 0u;
            if (blockIdx.x == 0) *(volatile unsigned long long *)(bar + (b + 1) % 3) = 0ull;
            const unsigned long long add = BAR_ONE + ((a & REQ) ? BAR_REQ : 0ull) + ((a & FAIL) ? BAR_ERR : 0ull);
            asm volatile("fence.acq_rel.gpu;\n\tred.release.gpu.global.add.u64 [%0], %1;"
                         ::"l"(bar + b % 3), "l"(add) : "memory");
        }
    }

    __device__ __forceinline__ unsigned wait()
    {
        if (threadIdx.x == 0) {
            unsigned long long v;
            unsigned it = 0, r = 0;
            for (;;) {
                asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(bar + b % 3) : "memory");
                if ((v & BAR_MASK) == gridDim.x) break;
                if (++it > spin) {
                    r = GAVE_UP;
                    break;
                }
                if (it > 64) __nanosleep(32);
            }
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
            if ((v / BAR_REQ) & BAR_MASK) r |= REQ;
            if (v / BAR_ERR) r |= FAIL;
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

// exclusive scan of the cell counts: segment g from the totals of the
// segments before it (the bin phase summed them) and its own counts
__device__ __forceinline__ void res_scan_seg(const ResArgs &A, int g, int nseg, int *wsum)
{
    constexpr int PER = RES_SEG / RES_BLOCK, NW = RES_BLOCK / 32;
    const int n = A.ncell, i0 = g * RES_SEG + threadIdx.x * PER;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int before = 0;
    for (int k = threadIdx.x; k < g; k += RES_BLOCK) before += A.segtot[k];
    int v[PER], own = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        v[k] = i0 + k < n ? A.ccount[i0 + k] : 0;
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
    if (g == nseg - 1 && threadIdx.x == RES_BLOCK - 1) A.cstart[n] = run;
    __syncthreads();
}

template <int N4>
__global__ void __launch_bounds__(RES_BLOCK, RES_MIN_BLOCKS) k_resident(const __grid_constant__ ResArgs A)
{
    __shared__ float dk[96];
    __shared__ unsigned acc_s[2], out_s;
    __shared__ int wsum[2 * (RES_BLOCK / 32)];
    step_block_setup(dk);
    const StepArgs &P = A.st;
    // no block writes the status words before every block has arrived at the last barrier
    const unsigned stop = *(volatile unsigned *)P.flags;
    bool rebuild = *((volatile unsigned *)P.flags + 1) != 0u;
    if (stop) return;                                         // a latched error stops the run
    if (threadIdx.x < 2) acc_s[threadIdx.x] = 0u;
    __syncthreads();
    if ((int)blockIdx.x == A.skip_block) return;              // barrier self-test: never arrives
    GridBar gb{A.bar, acc_s, &out_s, A.spin, 0};
    const int s = blockIdx.x * RES_BLOCK + threadIdx.x;
    const bool live = s < P.M;
    const int nseg = (A.ncell + RES_SEG - 1) / RES_SEG;
    const size_t Mp = (size_t)P.Mp;
    const int Mpi = P.Mp;
    const long long base = *(volatile long long *)P.stepp;    // the last step run

    int slot = 0, m = 0, cnt = 0;
    int4 bp = make_int4(-1, -1, -1, -1);
    float3 v = make_float3(0.f, 0.f, 0.f), d = v, gn = v;
    float4 rb = make_float4(0.f, 0.f, 0.f, 0.f), pi = rb;
    if (live) {
        slot = P.slot_of[s];
        m = melt_index(P, slot);
        bp = P.bp[s];
        cnt = P.nn[s];
        v = make_float3(P.u[s], P.u[Mpi + s], P.u[2 * Mpi + s]);
        const float4 d4 = A.dlt[A.cur0][s];
        d = make_float3(d4.x, d4.y, d4.z);
        rb = A.recb[s];
        pi = A.pg[A.cur0][s];
    }
    const MeltStep &md = P.melt[m];
    const float h = md.h, rc2 = P.rc2;
    const unsigned self = (unsigned)(live ? s : 0) | (13u << IDX_BITS);
    const unsigned *col = P.nl + (live ? s : 0);
    auto noise = [&](int it) {
        if (live)
            gn = gauss3_f(draw(P.seed, m, 0, (unsigned long long)(base + 1 + it), (uint32_t)(slot - md.off)));
    };
    noise(0);
    unsigned told = 0, builds = 0;
    for (int it = 0; it < A.K; ++it) {
        const int cur = A.cur0 ^ (it & 1);
        const float4 *pcur = A.pg[cur];
        if (rebuild) {                                        // Verlet rebuild; grid-uniform
            unsigned err = 0;
            if (live) {
                A.dlt[cur][s] = make_float4(d.x, d.y, d.z, 0.f);
                err = bin_md_one(*A.sim, s, A.x, A.xb64, A.recb, A.dlt[cur], A.pg[cur], nullptr, nullptr, A.cellid,
                                 A.rank, A.ccount, P.slot_of);
                if (err) atomicOr(A.errw, err);
                else {                                        // one atomic per segment and warp
                    const int g = A.cellid[s] / RES_SEG;
                    const unsigned act = __activemask(), grp = __match_any_sync(act, g);
                    if ((int)(threadIdx.x & 31) == __ffs(grp) - 1) atomicAdd(A.segtot + g, __popc(grp));
                }
            }
            gb.note(err ? FAIL : 0u);
            if ((told = gb.sync()) & (FAIL | GAVE_UP)) break;
            for (int g = blockIdx.x; g < nseg; g += gridDim.x) res_scan_seg(A, g, nseg, wsum);
            if ((told = gb.sync()) & GAVE_UP) break;
            if (live) scatter_one(s, A.cellid, A.rank, A.cstart, A.ctmp);
            if (blockIdx.x == 0)
                for (int g = threadIdx.x; g < nseg; g += RES_BLOCK) A.segtot[g] = 0;   // for the next rebuild
            if ((told = gb.sync()) & GAVE_UP) break;
            if (live && cellrank_one(s, A.cellid, A.cstart, A.ctmp, A.clist, A.recb, A.recs, A.ccount)) {
                atomicOr(A.errw, ERR_NL_CAPACITY);
                gb.note(FAIL);
            }
            if ((told = gb.sync()) & (FAIL | GAVE_UP)) break;
            err = nlist_masked<4>(A.nl, s, cnt);                 // whole warps; the row is read by its own thread only
            if (err) {
                atomicOr(A.errw, err);
                gb.note(FAIL);
            }
            d = make_float3(0.f, 0.f, 0.f);
            if (live) {
                rb = A.recb[s];
                pi = A.pg[cur][s];
            }
            ++builds;
        }
        unsigned err = 0;
        float3 F = make_float3(0.f, 0.f, 0.f);
        float4 part[4];
        part[0] = bp.x >= 0 ? pcur[bp.x] : pi;
        part[1] = bp.y >= 0 ? pcur[bp.y] : pi;
        part[2] = bp.z >= 0 ? pcur[bp.z] : pi;
        part[3] = bp.w >= 0 ? pcur[bp.w] : pi;
        const int kmax = __reduce_max_sync(0xffffffffu, cnt);
        for (int k0 = 0; k0 < kmax; k0 += RES_ILP) {
            unsigned e[RES_ILP];
            float4 pj[RES_ILP];
#pragma unroll
            for (int i = 0; i < RES_ILP; ++i) e[i] = k0 + i < cnt ? col[(size_t)(k0 + i) * Mp] : self;
#pragma unroll
            for (int i = 0; i < RES_ILP; ++i) pj[i] = pcur[e[i] & IDX_MASK];
#pragma unroll
            for (int i = 0; i < RES_ILP; ++i) {
                const unsigned q = e[i] >> IDX_BITS;
                const float dx = fmaf(dk[q], h, pj[i].x - pi.x);
                const float dy = fmaf(dk[32 + q], h, pj[i].y - pi.y);
                const float dz = fmaf(dk[64 + q], h, pj[i].z - pi.z);
                const float r2 = fmaf(dz, dz, fmaf(dy, dy, __fmul_rn(dx, dx)));
                float fr = mlj_fr32<N4>(P, r2);
                fr = (k0 + i < cnt && r2 < rc2) ? fr : 0.0f;
                F.x = fmaf(fr, dx, F.x); F.y = fmaf(fr, dy, F.y); F.z = fmaf(fr, dz, F.z);
            }
        }
        if (live) {
            bonded32<N4>(P, [&](int k, int) { return part[k]; }, md, pi, bp, F, err);
            v.x = fmaf(P.dt, fmaf(P.amp, gn.x, fmaf(-P.gamma, v.x, F.x)), v.x);
            v.y = fmaf(P.dt, fmaf(P.amp, gn.y, fmaf(-P.gamma, v.y, F.y)), v.y);
            v.z = fmaf(P.dt, fmaf(P.amp, gn.z, fmaf(-P.gamma, v.z, F.z)), v.z);
            d.x = fmaf(P.dt, v.x, d.x); d.y = fmaf(P.dt, v.y, d.y); d.z = fmaf(P.dt, v.z, d.z);
            pi = make_float4(rb.x + d.x, rb.y + d.y, rb.z + d.z, rb.w);
            A.pg[cur ^ 1][s] = pi;
            const bool far = fmaf(d.z, d.z, fmaf(d.y, d.y, __fmul_rn(d.x, d.x))) > P.half_skin2;
            if (!isfinite(v.x + v.y + v.z)) err |= ERR_NONFINITE;
            if (err) atomicOr(A.errw, err);
            gb.note((far ? REQ : 0u) | (err ? FAIL : 0u));
        }
        gb.arrive();
        if (it + 1 < A.K) noise(it + 1);
        told = gb.wait();
        rebuild = (told & REQ) != 0u;
        if (told & (FAIL | GAVE_UP)) break;
    }
    const int fin = A.cur0 ^ (A.K & 1);
    if (live) {
        A.dlt[fin][s] = make_float4(d.x, d.y, d.z, 0.f);
        P.u[s] = v.x; P.u[Mpi + s] = v.y; P.u[2 * Mpi + s] = v.z;
    }
    if (threadIdx.x == 0 && (told & GAVE_UP)) atomicOr(P.flags, ERR_TIMEOUT);
    if (blockIdx.x == 0 && threadIdx.x == 0) {                // every block has arrived at the last barrier
        if (told & FAIL) atomicOr(P.flags, *(volatile unsigned *)A.errw);
        P.flags[1] = rebuild ? 1u : 0u;
        P.flags[5] += builds;
        *A.stepp = base + A.K;
    }
}

template <int N4>
static cudaError_t launch_n4(const ResArgs &a, cudaStream_t st)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((a.st.M + RES_BLOCK - 1) / RES_BLOCK));
    cfg.blockDim = dim3(RES_BLOCK);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_resident<N4>, a);
}

static cudaError_t resident_start(int n4, const ResArgs &a, cudaStream_t st)
{
    switch (n4) {
        case 8: return launch_n4<8>(a, st);
        case 12: return launch_n4<12>(a, st);
        case 16: return launch_n4<16>(a, st);
        case 20: return launch_n4<20>(a, st);
        case 23: return launch_n4<23>(a, st);
        case 26: return launch_n4<26>(a, st);
        case 28: return launch_n4<28>(a, st);
        case 32: return launch_n4<32>(a, st);
        case 36: return launch_n4<36>(a, st);
        case 40: return launch_n4<40>(a, st);
        case 44: return launch_n4<44>(a, st);
        case 48: return launch_n4<48>(a, st);
        default: return launch_n4<0>(a, st);
    }
}

// One thread per monomer needs every block resident at once.
bool resident_fits(kg_ctx *c)
{
    if (c->precision != KG_MIXED || c->tpm != 1 || c->resident_failed) return false;
    if (c->res_blocks < 0) {
        int nsm = 0;
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, c->device);
        c->res_blocks = RES_MIN_BLOCKS * nsm;          // what __launch_bounds__ guarantees for every exponent
    }
    return (c->M + RES_BLOCK - 1) / RES_BLOCK <= c->res_blocks;
}

cudaError_t resident_launch(kg_ctx *c, int K, int skip_block, unsigned spin)
{
    ResArgs a{};
    a.st = step_args(c, c->cur);
    a.nl = nl_args(c);
    a.sim = c->d_sim;
    for (int b = 0; b < 2; ++b) {
        a.dlt[b] = c->dlt[b];
        a.pg[b] = c->pg[b];
    }
    a.x = c->x;
    a.xb64 = c->xb64;
    a.recb = c->recb;
    a.recs = c->recs;
    a.cellid = c->cellid;
    a.rank = c->rank;
    a.ccount = c->ccount;
    a.cstart = c->cstart;
    a.clist = c->clist;
    a.ctmp = c->ctmp;
    a.ncell = c->ncell_md;
    a.cur0 = c->cur;
    a.K = K;
    a.skip_block = skip_block;
    a.bar = c->resbar;
    a.errw = (unsigned *)(c->resbar + 3);
    a.segtot = (int *)(c->resbar + 4);
    a.spin = spin;
    a.stepp = c->d_step;
    // barrier words, error word and segment totals (a launch cut short leaves totals behind)
    const size_t nseg = (size_t)(c->ncell_md + RES_SEG - 1) / RES_SEG;
    cudaError_t e = cudaMemsetAsync(c->resbar, 0, 4 * sizeof(unsigned long long) + nseg * sizeof(int), c->stream);
    if (e != cudaSuccess) return e;
    e = resident_start(n4_of(c->stage.n), a, c->stream);
    if (e != cudaSuccess) return e;
    c->launches += 1;
    c->cur ^= K & 1;
    return cudaSuccess;
}

size_t resident_words(int ncell) { return 4 * sizeof(unsigned long long) + ((size_t)ncell / RES_SEG + 1) * sizeof(int); }

}  // namespace kg
