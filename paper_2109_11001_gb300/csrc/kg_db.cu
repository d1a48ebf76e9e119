// kg_db.cu -- double-bridging Monte Carlo sweep (Fig. 1; Sec. II.B criteria
// (i) and (ii)) with the semantics of a strictly sequential loop over attempts.
//
// A swap removes bond (A_p, A_{p+1}) and bond (B_q, B_{q+1}) of two chains and
// joins the ends crosswise so both chains keep N monomers:
//   kind 0 (q = p):      A' = A_0..A_p B_{p+1}..B_{N-1},  B' = B_0..B_p A_{p+1}..A_{N-1}
//   kind 1 (p+q = N-2):  A' = A_0..A_p B_q..B_0,          B' = A_{N-1}..A_{p+1} B_{q+1}..B_{N-1}
// (A the lower chain index).  Admissible iff both new and both removed bonds
// are <= 1.3 sigma.  Proposal: a bond drawn uniformly, then one entry of its
// partner list (ordered by monomer ids); acceptance
// min(1, exp(-dE/T) q(x'->x)/q(x->x')) with q ~ 1/|P(b1)| + 1/|P(b2)|.
//
// GPU organisation of one sweep:
//   1. bin every monomer on a grid of >= 1.3 sigma cells (positions do not move
//      during a sweep: swaps only relabel slots) and write its binary32 record
//      there; the 1.3 sigma criterion is decided on the records outside a
//      rounding band and in binary64 inside it, so decisions are exact;
//   2. k_db_eval: every attempt drawn in parallel against the pre-sweep
//      topology, one warp each (the 27 cells of a partner scan on its lanes):
//      its partner set and its partner.  A "monomer" here is its compute index;
//      the topology is the pair of maps slot -> monomer (comp_of) and monomer ->
//      slot (slot_of);
//   3. k_db_rounds (kg_db.cuh): drawn swaps are decided, and committed in order
//      in rounds: an attempt's record is stale when an earlier accepted swap in
//      the sweep touched one of its two chains, or put a junction monomer (whose
//      bonds changed) within one cell of a monomer whose neighbourhood it
//      scanned.  Nothing else an evaluation reads can change: swaps preserve
//      positions, the bonds inside moved segments, and the lengths of the two
//      pieces on either side of every bond;
//   4. k_db_finish: the box shifts are added to the positions in place; no
//      monomer data moves (the maps are the topology).
#include <cuda_runtime.h>

#include <algorithm>

#include "kg_db.cuh"

namespace kg {

// Attempt k: the drawn bond, its partner set and the partner drawn from it
// (one warp).  flags 0 (empty set, or a capacity error, which is flagged), or
// 1 | 4: to be decided from the parts below.
template <class V>
__device__ void draw_attempt(const DBC &C, const V &v, WarpCand &wc, unsigned long long seed, long long sweep, int k,
                             Attempt &a, unsigned &err)
{
    const MeltDev &md = C.md;
    const int N = md.N, off = md.off;
    a.flags = 0;
    a.d = -1;
    a.kind = a.A = a.B = a.pA = a.pB = a.q = 0;
    a.ver = 0;
    a.cell[2] = a.cell[3] = -1;
    a.p = a.dE = 0.0;
    const uint4 r = draw(seed, C.melt, 1, (unsigned long long)sweep, (uint32_t)k);
    const uint4 r2 = draw(seed, C.melt, 2, (unsigned long long)sweep, (uint32_t)k);
    const long long nbonds = (long long)md.n_ch * (N - 1);
    const long long bond = mul_hi64(((unsigned long long)r.y << 32) | r.x, (unsigned long long)nbonds);
    const int c = (int)(bond / (N - 1)), b = (int)(bond % (N - 1));
    a.c = c;
    a.cell[0] = C.cell[v.occ(off + c * N + b)];
    a.cell[1] = C.cell[v.occ(off + c * N + b + 1)];
    a.n = warp_partners<true>(C, v, c, b, wc, err);
    if (a.n <= 0) return;
    const Cand m = wc.cand[mul_hi64(((unsigned long long)r2.y << 32) | r2.x, (unsigned long long)a.n)];
    a.flags = 1 | 4;
    a.d = m.d;
    a.q = m.q;
    a.cell[2] = C.cell[v.occ(off + m.d * N + m.q)];
    a.cell[3] = C.cell[v.occ(off + m.d * N + m.q + 1)];
    a.kind = m.kind;
    a.A = c < m.d ? c : m.d;
    a.B = c < m.d ? m.d : c;
    a.pA = a.A == c ? b : m.q;
    a.pB = a.A == c ? m.q : b;
}

// Part t of deciding a drawn swap (one warp): the sizes of the partner sets of
// the partner bond and, in the topology after the swap, of both new bonds, and
// the energy change.
constexpr int UNIFORM_TASKS = 4;

template <class V>
__device__ double swap_part(const DBC &C, const V &v, WarpCand &wc, const Attempt &a, int t, unsigned &err)
{
    const int lane = threadIdx.x & 31;
    const ViewMove<V> w{v, a.kind, a.A, a.B, a.pA, a.pB, C.md.N, C.md.off};
    if (t < 3) {
        const int n = t == 0 ? warp_partners<false>(C, v, a.d, a.q, wc, err)
                             : warp_partners<false>(C, w, t == 1 ? a.A : a.B, t == 1 ? a.pA : a.pB, wc, err);
        if (n <= 0) err |= n < 0 ? ERR_DB_CAPACITY : ERR_DB_INTERNAL;
        return (double)n;
    }
    // dE: a lane per term (a binary64 square root, divide or logarithm is a long
    // dependent chain), the sum in the order new bonds, old bonds, new angles, old angles
    double term = 0.0;
    if (lane < 4) {
        term = bond_fene(C, ViewEither<V>{w, lane < 2}, lane & 1 ? a.B : a.A, lane & 1 ? a.pB : a.pA);
    } else if (lane < 12) {
        const int i = lane & 3;
        term = bend(C, ViewEither<V>{w, lane < 8}, i < 2 ? a.A : a.B, (i < 2 ? a.pA : a.pB) + (i & 1));
    }
    auto at = [&](int k) { return __shfl_sync(FULL_MASK, term, k); };
    double dE = at(0) + at(1) - at(2) - at(3);
    dE += at(4) + at(5) + at(6) + at(7);
    dE -= at(8) + at(9) + at(10) + at(11);
    return dE;
}

constexpr int EVAL_WARPS_U = 4;                 // attempts (warps) per block of k_db_eval

// (128, 12): at most 40 registers; the partner scans are latency-bound, and
// more resident warps beat the spills (160,000 attempts: 157 us)
__global__ void __launch_bounds__(32 * EVAL_WARPS_U, 12) k_db_eval(const SimDev *__restrict__ Sp,
                                                              const StageDev *__restrict__ stp,
                                                              const double *__restrict__ x,
                                                              const int *__restrict__ pid,
                                                              const int *__restrict__ cell,
                                                              const int *__restrict__ start,
                                                              const int *__restrict__ list,
                                                              const float4 *__restrict__ rec,
                                                              const int *__restrict__ koff,
                                                              const int *__restrict__ comp_of,
                                                              const int *__restrict__ slot_of,
                                                              Attempt *__restrict__ att, long long sweep,
                                                              unsigned *flags)
{
    __shared__ WarpCand wcs[EVAL_WARPS_U];
    if (flags[0]) return;                          // a latched error stops the sweep (no block barrier follows)
    const SimDev &S = *Sp;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = blockIdx.x * EVAL_WARPS_U + warp;
    if (g >= koff[S.n_melts]) return;
    int m = 0;
    while (g >= koff[m + 1]) ++m;
    const DBC C = make_dbc(S, *stp, m, x, pid, cell, start, list, rec, stp->T);
    unsigned err = 0;
    Attempt a;
    draw_attempt(C, ViewMap{comp_of, slot_of}, wcs[warp], S.seed, sweep, g - koff[m], a, err);
    if (lane == 0) {
        att[g] = a;
        if (err) atomicOr(flags, err);
    }
}

// uniform proposal: a stale record is re-evaluated by one warp; the
// staleness radius is one cell
struct UniformEval {
    const SimDev *S;
    const StageDev *st;
    const double *x;
    const int *pid, *cell, *start, *list;
    const float4 *rec;
    const int *comp_of, *slot_of;
    long long sweep;
    unsigned *errw;              // RoundArgs::errw
    WarpCand *wc;                // set by the kernel
    static constexpr int TASKS = UNIFORM_TASKS;
    __device__ DBC dbc(int m) const { return make_dbc(*S, *st, m, x, pid, cell, start, list, rec, st->T); }
    __device__ void say(unsigned err) const
    {
        if (err && (threadIdx.x & 31) == 0) atomicOr(errw, err);
    }
    __device__ void scan(int m, int k, int, Attempt &a)
    {
        unsigned err = 0;
        draw_attempt(dbc(m), ViewMap{comp_of, slot_of}, *wc, S->seed, sweep, k, a, err);
        say(err);
    }
    __device__ double task(int m, const Attempt &a, int t)
    {
        unsigned err = 0;
        const double v = swap_part(dbc(m), ViewMap{comp_of, slot_of}, *wc, a, t, err);
        say(err);
        return v;
    }
    __device__ bool accepts(int m, int k, const Attempt &a, const double *p) const
    {
        if (!(p[0] > 0.0 && p[1] > 0.0 && p[2] > 0.0)) return false;     // an error, flagged
        double acc = exp(-p[3] / st->T);
        if (!S->paper_metropolis) acc *= (1.0 / p[1] + 1.0 / p[2]) / (1.0 / a.n + 1.0 / p[0]);
        return accept_u(S->seed, m, sweep, k) < acc;
    }
};

struct UniformRadius {
    __device__ int radius(const MeltDev &) const { return 1; }
};

constexpr int ROUND_WARPS = 8;

// (256, 3): three records' checks and evaluations per scheduler in flight hide more than the registers cost
__global__ void __launch_bounds__(32 * ROUND_WARPS, 3) k_db_rounds(RoundArgs R, UniformEval ev)
{
    __shared__ WarpCand wcs[ROUND_WARPS];
    ev.wc = wcs + (threadIdx.x >> 5);
    UniformRadius pol;
    rounds_body<32 * ROUND_WARPS>(ev, pol, R);
}

// end of a sweep: box shifts into the positions (x + L*img, as one rounding of
// a product and one of a sum), counters cleared
__global__ void __launch_bounds__(256) k_db_finish(const SimDev *__restrict__ Sp, double *__restrict__ x,
                                                  const int *__restrict__ slot_of, int *__restrict__ img,
                                                  double *__restrict__ msd_ref, double *__restrict__ xb64)
{
    const SimDev &S = *Sp;
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= S.M) return;
    const int Mp = S.Mp;
    const double L = S.melt[melt_of(S, slot_of[j])].L;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int k = img[d * Mp + j];
        if (k) {
            x[d * Mp + j] = __dadd_rn(x[d * Mp + j], __dmul_rn(L, (double)k));
            if (msd_ref) msd_ref[d * Mp + j] = __dadd_rn(msd_ref[d * Mp + j], __dmul_rn(L, (double)k));
            if (xb64) xb64[d * Mp + j] = __dadd_rn(xb64[d * Mp + j], __dmul_rn(L, (double)k));
        }
        img[d * Mp + j] = 0;
    }
}

// kg_md.cu
__global__ void k_bin_db(const SimDev *__restrict__ Sp, const double *__restrict__ x, int *__restrict__ cellid,
                         int *__restrict__ rank, int *__restrict__ count, const int *__restrict__ slot_of,
                         float4 *__restrict__ rec);
__global__ void k_scan1(const int *__restrict__ in, int *__restrict__ out, int *__restrict__ bsum, int n,
                        const unsigned *__restrict__ flags);
__global__ void k_scan2(int *__restrict__ out, const int *__restrict__ bsum, int n, int nblk,
                        const unsigned *__restrict__ flags);
__global__ void k_scatter(const int *__restrict__ cellid, const int *__restrict__ rank,
                          const int *__restrict__ start, int *__restrict__ list, int M,
                          const unsigned *__restrict__ flags);

static inline int nblk(long long n, int b) { return (int)((n + b - 1) / b); }

void db_bin(kg_ctx *c, const std::vector<long long> &K)
{
    cudaStream_t st = c->stream;
    const int nm = c->sim.n_melts;
    c->launches += 5;
    std::vector<int> koff(nm + 1, 0);
    for (int m = 0; m < nm; ++m) koff[m + 1] = koff[m] + (int)K[m];
    cudaMemcpyAsync(c->koff, koff.data(), sizeof(int) * (nm + 1), cudaMemcpyHostToDevice, st);
    // grid of >= 1.3 sigma cells
    cudaMemsetAsync(c->dbcount, 0, sizeof(int) * c->ncell_db, st);
    k_bin_db<<<nblk(c->M, 256), 256, 0, st>>>(c->d_sim, c->x, c->dbcell, c->dbrank, c->dbcount, c->slot_of,
                                              c->dbrec);
    const int nb = nblk(c->ncell_db, 1024);
    k_scan1<<<nb, 1024, 0, st>>>(c->dbcount, c->dbstart, c->bsum, c->ncell_db, nullptr);
    k_scan2<<<nb, 1024, 0, st>>>(c->dbstart, c->bsum, c->ncell_db, nb, nullptr);
    k_scatter<<<nblk(c->M, 256), 256, 0, st>>>(c->dbcell, c->dbrank, c->dbstart, c->dblist, c->M, nullptr);
}

void db_finish(kg_ctx *c, long long *host_stats)
{
    cudaStream_t st = c->stream;
    c->launches += 1;
    // box shifts into the positions; chain partners follow the new maps
    k_db_finish<<<nblk(c->M, 256), 256, 0, st>>>(c->d_sim, c->x, c->slot_of, c->img, c->msd_ref, c->xb64);
    bonded_partners(c);
    cudaMemcpyAsync(host_stats, c->db_stats, sizeof(long long) * 4 * c->sim.n_melts, cudaMemcpyDeviceToHost, st);
}

void db_rounds_reset(kg_ctx *c)
{
    cudaStream_t st = c->stream;
    cudaMemsetAsync(c->chain_ver, 0xFF, sizeof(int) * (size_t)c->n_chain_total, st);    // -1: untouched
    cudaMemsetAsync(c->dbmark, 0xFF, sizeof(int) * (size_t)c->ncell_db, st);
    std::vector<int> r0((size_t)2 * RS * MAX_MELTS, 0);
    for (int m = 0; m < 2 * MAX_MELTS; ++m) r0[(size_t)RS * m + 4] = INT_MAX;   // no accepted attempt known
    cudaMemcpyAsync(c->dbround, r0.data(), sizeof(int) * r0.size(), cudaMemcpyHostToDevice, st);
}

RoundArgs round_args(kg_ctx *c)
{
    RoundArgs r{};
    r.sim = c->d_sim;
    r.x = c->x;
    r.cell = c->dbcell;
    r.koff = c->koff;
    r.att = (Attempt *)c->att;
    r.occ = c->comp_of;
    r.curmap = c->slot_of;
    r.img = c->img;
    r.chain_ver = c->chain_ver;
    r.cell_ver = c->dbmark;
    r.round = c->dbround;
    r.old = (int *)c->scratch;
    r.stats = c->db_stats;
    r.flags = c->flags;
    r.errw = (unsigned *)(c->dbbar + 3);
    return r;
}

cudaError_t db_sweep(kg_ctx *c, const std::vector<long long> &K, long long *host_stats)
{
    cudaStream_t st = c->stream;
    const int nm = c->sim.n_melts;
    long long tot = 0;
    for (long long k : K) tot += k;
    db_bin(c, K);
    // speculative evaluation
    Attempt *att = (Attempt *)c->att;
    if (tot > 0)
        k_db_eval<<<nblk(tot, EVAL_WARPS_U), 32 * EVAL_WARPS_U, 0, st>>>(
            c->d_sim, c->d_stage, c->x, c->pid, c->dbcell, c->dbstart, c->dblist, c->dbrec, c->koff, c->comp_of,
            c->slot_of, att, c->sweep, c->flags);
    // ordered commit in rounds (kg_db.cuh)
    db_rounds_reset(c);
    const RoundArgs ra = round_args(c);
    const UniformEval ev{c->d_sim, c->d_stage, c->x, c->pid, c->dbcell, c->dbstart, c->dblist, c->dbrec,
                         c->comp_of, c->slot_of, c->sweep, ra.errw, nullptr};
    const cudaError_t e = rounds_launch(c, k_db_rounds, 32 * ROUND_WARPS, 0, tot, nm, ra, ev);
    if (e != cudaSuccess) return e;
    c->launches += 1;
    db_finish(c, host_stats);
    return cudaSuccess;
}

}  // namespace kg
