// kg_resident.cu -- the mixed path's MD loop for systems whose monomers all fit
// the GPU's resident threads: one cooperative launch runs K steps, one thread
// per monomer.
//
// What bounds a small system is not work but the chain of dependent waits: as
// separate launches a step was a begin kernel, a conditional graph node and a
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
// Every wait is bounded by a poll count (2^22 of 0.32 us, 1.3 s), after which the
// block latches ERR_TIMEOUT and leaves; the grid itself starts when all its
// blocks fit, so a busy GPU uses up no polls.  The arithmetic is that of the one-step kernel
// (kg_step.cuh) on the same lists, so trajectories have the same bits.
//
// Measured, 50 steps and a read of the state of 80,000 monomers (skin 0.3, n =
// 12, dt = 0.01; a build every third or fourth step), against captured graphs
// of separate launches: 1748 -> 1090 us.
// Larger systems go in whole tiles (kg_resident_tiled.cu) or, from 1280
// monomers per SM, through the captured loop (kg_md.cu).
//
// Systems of at most 128 monomers per SM take kg_resident_small.cu.
//
// (128, 5): at most 102 registers, 5 x 128 threads per SM, about 97,000
// monomers on 152 SMs (resident_kind).
#include <cuda_runtime.h>

#include <algorithm>

#include "kg_resident.cuh"

namespace kg {

constexpr int RES_BLOCK = 128;
constexpr int RES_MIN_BLOCKS = 5;
constexpr int RES_ILP = 8;               // list entries in flight per lane

template <int N4>
__global__ void __launch_bounds__(RES_BLOCK, RES_MIN_BLOCKS) k_resident(const __grid_constant__ ResArgs A)
{
    __shared__ float dk[96];
    __shared__ unsigned acc_s[2], out_s;
    __shared__ int wsum[RES_BLOCK / 16];
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
                err = bin_md_one(*A.sim, s, A.x, A.xb64, A.recb, A.dlt[cur], A.dlt[cur], A.pg[cur], nullptr, nullptr, A.cellid,
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
            for (int g = blockIdx.x; g < nseg; g += gridDim.x) res_scan_seg<RES_BLOCK>(A, A.ccount, g, nseg, wsum);
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
            bonded32<N4>(P, [&](int k, int) { return part[k]; }, [&](int, float a, float3 x) { axpy3(a, x, F); }, md,
                         pi, bp, err);
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
        if (builds) P.flags[RES_BUILT] = 0u;                  // the cell order is in clist
        *A.stepp = base + A.K;
    }
}

// How a context's steps run: RES_NONE (launches per step), RES_WIDE (this
// file's kernel, 640 monomers per SM), RES_SMALL (kg_resident_small.cu, 128
// monomers per SM) or RES_TILED (kg_resident_tiled.cu, any number; by default
// while a block has one tile of 256).  Every block has to be resident at once;
// the limits are what the kernels' __launch_bounds__ guarantee for every
// exponent.
//
// Dilute systems: a list build scans every cell, here from a block per 64 to
// 256 monomers, there from the whole GPU.  At 85 to 90 cells per monomer the
// resident loops are still ahead (us per step against the captured loop; 1,000
// monomers 7.8 / 9.4, 19,000 9.5 / 14.1, 90,000 17.3 / 31.2), the work per
// block grows with the cells, and no use of so empty a box is known, so the
// rule ends there.
constexpr int TILED_MOST = 5 * 256;
constexpr long long DILUTE_CELLS = 64;           // cells per monomer

int resident_kind(kg_ctx *c)
{
    if (c->res_sms < 0) cudaDeviceGetAttribute(&c->res_sms, cudaDevAttrMultiProcessorCount, c->device);
    if (c->precision != KG_MIXED || c->resident_failed) return RES_NONE;
    if (c->tpm != 1 && !(c->p.flags & KG_FLAG_PERSISTENT)) return RES_NONE;
    if (c->ncell_md > DILUTE_CELLS * c->M + 4096) return c->p.flags & KG_FLAG_PERSISTENT ? RES_TILED : RES_NONE;
    if (c->buckets && c->M <= SMALL_OWN * SMALL_MIN_BLOCKS * c->res_sms) return RES_SMALL;
    if (c->M <= RES_BLOCK * RES_MIN_BLOCKS * c->res_sms) return RES_WIDE;
    return c->M <= TILED_MOST * c->res_sms || (c->p.flags & KG_FLAG_PERSISTENT) ? RES_TILED : RES_NONE;
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
        a.count[b] = c->bcount ? c->bcount + (size_t)b * c->ncell_md : nullptr;
    }
    a.bidx = c->bidx;
    a.brec = c->brec;
    a.brec2 = c->brec ? c->brec + (size_t)c->ncell_md * BUCKET_MAIN : nullptr;
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
    const int n4 = n4_of(c->stage.n), nb = (c->M + RES_BLOCK - 1) / RES_BLOCK;
    const int kind = resident_kind(c);
    e = kind == RES_SMALL  ? small_launch(a, n4, c->stream)
        : kind == RES_WIDE ? KG_RESIDENT_LAUNCH(k_resident, n4, nb, RES_BLOCK, a, c->stream)
                           : tiled_launch(a, n4, c->res_sms, c->stream);
    if (e != cudaSuccess) return e;
    c->launches += 1;
    c->cur ^= K & 1;
    return cudaSuccess;
}

// Barrier words and segment totals; for the small kernel bucket counts (two
// sets), members and records, 648 bytes a cell.  Cells of the usual grids hold
// 2.4 to 5 monomers; grids whose mean is above a third of a bucket (cell_scale
// well above 1) do not use them, nor do those with more than eight cells per
// monomer: a thousand monomers in a box of side 500 have 44 million cells.  At
// the limit the buckets of 19,000 monomers take 100 MB (one thread per monomer
// without them: 7.4 against 6.0 us per step there).
constexpr long long BUCKET_CELLS = 8;            // cells per monomer

bool resident_alloc(kg_ctx *c)
{
    double most = 0.0;
    for (int m = 0; m < c->sim.n_melts; ++m) {
        const MeltDev &md = c->sim.melt[m];
        most = std::max(most, (double)md.M / ((double)md.nc * md.nc * md.nc));
    }
    c->buckets = 3.0 * most <= BUCKET && c->ncell_md <= BUCKET_CELLS * c->M + 512;
    const int kind = resident_kind(c);
    if (c->precision != KG_MIXED) return true;
    c->resbar = (unsigned long long *)dev_alloc(c, 4 * sizeof(unsigned long long) +
                                                       ((size_t)c->ncell_md / RES_SEG + 1) * sizeof(int));
    if (kind != RES_SMALL) return c->resbar != nullptr;
    const size_t nb = (size_t)c->ncell_md * BUCKET;
    c->bcount = (int *)dev_alloc(c, 2 * (size_t)c->ncell_md * sizeof(int));
    c->bidx = (int *)dev_alloc(c, nb * sizeof(int));
    c->brec = (float4 *)dev_alloc(c, nb * sizeof(float4));
    return c->resbar && c->bcount && c->bidx && c->brec;
}

// a rebuild cut short by an error may have left counts behind (kg_load_config)
cudaError_t resident_reset(kg_ctx *c)
{
    return c->bcount ? cudaMemsetAsync(c->bcount, 0, 2 * sizeof(int) * (size_t)c->ncell_md, c->stream) : cudaSuccess;
}

// The cell order of a build that used buckets, for a re-sort: the counts to
// the counting sort's array for the scan, then every bucket's members (in
// order, from the records) to their cell's run.
__global__ void __launch_bounds__(256) k_bucket_counts(const unsigned *__restrict__ flags,
                                                      const int *__restrict__ bcount, int ncell,
                                                      int *__restrict__ count)
{
    const unsigned built = flags[RES_BUILT];
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (built && c < ncell) count[c] = bcount[(size_t)(built - 1) * ncell + c];
}

__global__ void __launch_bounds__(256) k_bucket_list(const unsigned *__restrict__ flags,
                                                    const float4 *__restrict__ brec, int ncell,
                                                    int *__restrict__ count, const int *__restrict__ start,
                                                    int *__restrict__ list)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (!flags[RES_BUILT] || c >= ncell) return;
    const int n = count[c], k0 = start[c];
    for (int k = 0; k < n; ++k) list[k0 + k] = __float_as_int(
            (k < BUCKET_MAIN ? brec[(size_t)c * BUCKET_MAIN + k]
                             : brec[(size_t)ncell * BUCKET_MAIN + (size_t)c * (BUCKET - BUCKET_MAIN) + k - BUCKET_MAIN])
                .w);
    count[c] = 0;
}

void resident_cell_order(kg_ctx *c)
{
    if (!c->bcount) return;
    const int nb = (c->ncell_md + 255) / 256;
    k_bucket_counts<<<nb, 256, 0, c->stream>>>(c->flags, c->bcount, c->ncell_md, c->ccount);
    scan_counts(c, c->ccount, c->cstart, c->ncell_md, c->bsum);
    k_bucket_list<<<nb, 256, 0, c->stream>>>(c->flags, c->brec, c->ncell_md, c->ccount, c->cstart, c->clist);
    c->launches += 4;
}

}  // namespace kg
