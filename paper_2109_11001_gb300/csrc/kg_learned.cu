// kg_learned.cu -- double-bridging sweep with a learned partner proposal.
//
// The paper draws a swap partner uniformly from the admissible list P(b) of
// the drawn bond (Fig. 1).  Here the list, in the same order, is weighted by
//     pi_j = (1 - lambda) softmax_j(s) + lambda / |P(b)|,
// s_j the logit the network (kg_mlp.cuh) assigns to the features of swap j,
// and the swap is accepted with min(1, exp(-dE/T) q(x'->x) / q(x->x')), where
// q(x->x') = pi_b(move) + pi_b'(move) sums the two ways of proposing it (either
// removed bond drawn) and q(x'->x) the same in the swapped state.  lambda > 0
// keeps every admissible swap proposable, so the chain stays irreducible;
// lambda = 1 is the uniform proposal, with the Hastings ratio of Fig. 1.
//
// Features (24 per swap; u-w the drawn bond, X-Y the partner bond, new bonds
// u-X and Y-w; every value depends on positions and bonds only, not on the
// direction in which a chain's slots are numbered):
//   0-1 removed bond lengths (sorted)       2-3 new bond lengths (sorted)
//   4   change of the FENE terms             5   change of the bending energy
//   6-9 cos at the four junction vertices, before (sorted)
//   10-13 the same after                    14-17 cos one vertex further out (sorted)
//   18  cos between u->w and X->Y            19 kappa/4   20 n/12
//   21  min(p+1, N-1-p)/N (p the drawn bond) 22 dE = 4 + 5   23 1
//
// GPU organisation (one warp per attempt): the warp scans the 27 cells around
// the drawn bond's lower monomer, ranks the candidates by monomer ids, computes
// their features (FP64, one lane each), runs the network on the tensor cores
// in 16-row tiles, and lane 0 forms pi in FP64 in list order.  The forward
// probability of the partner bond and the two reverse probabilities repeat
// this for three more bonds (the reverse ones in the swapped topology view).
// Attempts are drawn speculatively in parallel, then decided and committed in
// order by the shared commit rounds (kg_db.cuh); a learned evaluation reads monomers up
// to 2 b_lim + 3 b_max from its junction monomers (b_lim = 1.3 the swap bond
// limit, b_max the longest bond at sweep start), so an accepted swap with a
// junction monomer within that many cells forces a re-evaluation.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "kg_db.cuh"
#include "kg_mlp.cuh"

namespace kg {

struct LearnedArgs {
    double lambda;
    const MlpSmem *w;                   // bf16 image of the network
    double *logf, *logt;                // per-attempt log staging (null: no log)
    int *logn;
    const unsigned long long *bmax2;    // longest bond squared, binary64 bits
    const float4 *rec;                  // binary32 records on the DB grid (swap-bond prefilter)
};

// per-warp shared scratch of one proposal evaluation
struct __align__(16) WarpProp : WarpCand {
    double pi[CAND_CAP];
    double dE[CAND_CAP];
    float s[CAND_CAP];
    double f[24];                       // features of the candidate in work
    __nv_bfloat16 F[CAND_CAP * S1];     // features of the candidates, bf16 rows
};

constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ void sort4(double *v)
{
    for (int i = 1; i < 4; ++i) {
        const double t = v[i];
        int j = i - 1;
        while (j >= 0 && v[j] > t) {
            v[j + 1] = v[j];
            --j;
        }
        v[j + 1] = t;
    }
}

// Features of swap m of bond (c, b) in view v into f (shared), whole warp: a
// lane per bond length and per cosine (each a dependent chain of binary64
// square roots and divides), then lane 0 sorts and sums them.
template <class V>
__device__ void move_features(const DBC &C, const V &v, int c, int b, const Cand &m, double *f)
{
    const int lane = threadIdx.x & 31;
    const MeltDev &md = C.md;
    const int N = md.N, off = md.off;
    const int u = v.occ(off + c * N + b), w = v.occ(off + c * N + b + 1);
    int X, Y;
    if (m.kind == 0) {
        Y = v.occ(off + m.d * N + b);
        X = v.occ(off + m.d * N + b + 1);
    } else {
        X = v.occ(off + m.d * N + m.q);
        Y = v.occ(off + m.d * N + m.q + 1);
    }
    const int A = c < m.d ? c : m.d, B = c < m.d ? m.d : c;
    const int pA = A == c ? b : m.q, pB = A == c ? m.q : b;
    // lanes 0-3: lengths of u-w, X-Y, u-X, Y-w and their FENE terms; 4-7, 8-11,
    // 12-15: cosines at the four junction vertices before and after, and one
    // vertex further out; 16: cosine between u->w and X->Y
    double val = 0.0, fene = 0.0;
    if (lane < 4) {
        val = sqrt(d2(C, lane & 1 ? (lane == 1 ? X : Y) : u, lane == 0 || lane == 3 ? w : (lane == 1 ? Y : X)));
        fene = fene_of_r(C, val);
    } else if (lane < 16) {
        const int t = lane & 3, far = lane >= 12 ? ((t & 1) ? 1 : -1) : 0;
        const ViewEither<V> e{ViewMove<V>{v, m.kind, A, B, pA, pB, N, off}, lane >= 8 && lane < 12};
        val = vcos(C, e, t < 2 ? A : B, (t < 2 ? pA : pB) + (t & 1) + far);
    } else if (lane == 16) {
        double e1[3], e2[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            e1[k] = min_image_exact(C.x[k * C.Mp + w] - C.x[k * C.Mp + u], md.L, md.invLf);
            e2[k] = min_image_exact(C.x[k * C.Mp + Y] - C.x[k * C.Mp + X], md.L, md.invLf);
        }
        val = (e1[0] * e2[0] + e1[1] * e2[1] + e1[2] * e2[2])
              / (sqrt(e1[0] * e1[0] + e1[1] * e1[1] + e1[2] * e1[2]) *
                 sqrt(e2[0] * e2[0] + e2[1] * e2[1] + e2[2] * e2[2]));
    }
    auto at = [&](int k) { return __shfl_sync(FULL, val, k); };
    const double o1 = at(0), o2 = at(1), n1 = at(2), n2 = at(3);
    double before[4] = {at(4), at(5), at(6), at(7)}, after[4] = {at(8), at(9), at(10), at(11)};
    double outer[4] = {at(12), at(13), at(14), at(15)};
    const double cross = at(16);
    const double fo1 = __shfl_sync(FULL, fene, 0), fo2 = __shfl_sync(FULL, fene, 1);
    const double fn1 = __shfl_sync(FULL, fene, 2), fn2 = __shfl_sync(FULL, fene, 3);
    if (lane == 0) {
        f[0] = o1 < o2 ? o1 : o2;
        f[1] = o1 < o2 ? o2 : o1;
        f[2] = n1 < n2 ? n1 : n2;
        f[3] = n1 < n2 ? n2 : n1;
        f[4] = fn1 + fn2 - fo1 - fo2;
        double db = 0.0;
#pragma unroll
        for (int i = 0; i < 4; ++i) db += md.kappa * ((1.0 - after[i]) - (1.0 - before[i]));
        f[5] = db;
        sort4(before);
        sort4(after);
        sort4(outer);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            f[6 + i] = before[i];
            f[10 + i] = after[i];
            f[14 + i] = outer[i];
        }
        f[18] = cross;
        f[19] = md.kappa / 4.0;
        f[20] = C.nexp / 12.0;
        const int lo = b + 1 < N - 1 - b ? b + 1 : N - 1 - b;
        f[21] = (double)lo / N;
        f[22] = f[4] + f[5];
        f[23] = 1.0;
    }
    __syncwarp();
}

// Proposal weights of bond (c, b) in view v: wp.cand[0..n), wp.pi, and (when
// `features` or the network is in use) wp.dE and wp.F; wp.s (the logits) when
// the network ran (lambda < 1 and n > 1, or `logits`).  log_att >= 0 writes the
// FP64 features and targets min(1, exp(-dE/T)) of every candidate to that
// attempt's log rows.  Returns n (0: empty, -1: capacity error).
template <class V>
__device__ int proposal(const DBC &C, const V &v, const MlpSmem &W, WarpProp &wp, const LearnedArgs &la, int c,
                        int b, bool features, long long log_att, unsigned &err, bool logits = false)
{
    const int lane = threadIdx.x & 31;
    const int n = warp_partners<true>(C, v, c, b, wp, err);
    if (n <= 0) return n;
    // A one-entry list proposes its only swap with pi = (1 - lambda) + lambda
    // whatever the logit (the softmax of one value is exactly 1, so pi has the
    // same bits either way): unless the caller wants the logits, the network
    // and, unless dE or the log needs them, the features are skipped
    const bool net = la.lambda < 1.0 && (n > 1 || logits);
    if (net || features) {
        const int nr = (n + 15) & ~15;
        for (int j = 0; j < n; ++j) {                  // most lists have one entry
            move_features(C, v, c, b, wp.cand[j], wp.f);
            __nv_bfloat16 *row = wp.F + j * S1;
            row[lane] = lane < 24 ? __double2bfloat16(wp.f[lane]) : __float2bfloat16(0.f);
            if (log_att >= 0 && lane < 24) la.logf[(log_att * CAND_CAP + j) * 24 + lane] = wp.f[lane];
            if (lane == 0) {
                wp.dE[j] = wp.f[22];
                if (log_att >= 0) {
                    const double de = wp.f[22] / C.T;
                    la.logt[log_att * CAND_CAP + j] = de > 0.0 ? exp(-de) : 1.0;
                }
            }
            __syncwarp();
        }
        for (int j = n; j < nr; ++j) wp.F[j * S1 + lane] = __float2bfloat16(0.f);
        if (log_att >= 0 && lane == 0) la.logn[log_att] = n;
        __syncwarp();
    }
    if (net) {
        const int g = lane >> 2;
        for (int r0 = 0; r0 < n; r0 += 16) {
            float s0, s1;
            mlp_forward16(W, wp.F + r0 * S1, s0, s1);
            if ((lane & 3) == 0) {
                if (r0 + g < n) wp.s[r0 + g] = s0;
                if (r0 + g + 8 < n) wp.s[r0 + g + 8] = s1;
            }
        }
        __syncwarp();
    }
    if (lane == 0) {                                // FP64, in list order
        double smax = -1e300, z = 0.0;
        for (int j = 0; j < n; ++j) {
            const double s = net ? (double)wp.s[j] : 0.0;
            if (s > smax) smax = s;
        }
        for (int j = 0; j < n; ++j) z += exp((net ? (double)wp.s[j] : 0.0) - smax);
        for (int j = 0; j < n; ++j)
            wp.pi[j] = (1.0 - la.lambda) * exp((net ? (double)wp.s[j] : 0.0) - smax) / z + la.lambda / n;
    }
    __syncwarp();
    return n;
}

// Probability that bond (c, b)'s proposal picks the swap (kind, A, B, pA, pB).
template <class V>
__device__ double match_prob(const DBC &C, const V &v, const MlpSmem &W, WarpProp &wp, const LearnedArgs &la,
                             int c, int b, int kind, int A, int B, int pA, int pB, unsigned &err)
{
    const int lane = threadIdx.x & 31;
    const int n = proposal(C, v, W, wp, la, c, b, false, -1, err);
    double p = 0.0;
    if (n > 0 && lane == 0) {
        for (int j = 0; j < n; ++j) {
            const Cand &m = wp.cand[j];
            const int a2 = c < m.d ? c : m.d, b2 = c < m.d ? m.d : c;
            const int pa2 = a2 == c ? b : m.q, pb2 = a2 == c ? m.q : b;
            if (m.kind == kind && a2 == A && b2 == B && pa2 == pA && pb2 == pB) {
                p = wp.pi[j];
                break;
            }
        }
    }
    p = __shfl_sync(FULL, p, 0);
    __syncwarp();
    return p;
}

// Attempt k of this melt's sweep (g its global index): the drawn bond, its
// proposal and the partner picked from it (one warp).  flags 0 (empty set, or a
// capacity error, which is flagged), or 1 | 4: to be decided from the parts.
template <class V>
__device__ void learned_draw(const DBC &C, const V &v, const MlpSmem &W, WarpProp &wp, const LearnedArgs &la,
                             unsigned long long seed, long long sweep, int k, int g, Attempt &a, unsigned &err)
{
    const int lane = threadIdx.x & 31;
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
    const double upick = (double)((((unsigned long long)r2.y << 32) | r2.x) >> 11) * (1.0 / 9007199254740992.0);
    const int c = (int)(bond / (N - 1)), b = (int)(bond % (N - 1));
    a.c = c;
    a.cell[0] = C.cell[v.occ(off + c * N + b)];
    a.cell[1] = C.cell[v.occ(off + c * N + b + 1)];
    if (la.logn && lane == 0) la.logn[g] = 0;
    a.n = proposal(C, v, W, wp, la, c, b, true, la.logf ? (long long)g : -1LL, err);
    if (a.n <= 0) return;
    int j = 0;
    if (lane == 0) {
        double cum = wp.pi[0];
        while (j + 1 < a.n && upick >= cum) cum += wp.pi[++j];
    }
    j = __shfl_sync(FULL, j, 0);
    const Cand m = wp.cand[j];
    a.p = wp.pi[j];
    a.dE = wp.dE[j];
    __syncwarp();
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

constexpr int EVAL_WARPS = 4;

__host__ __device__ constexpr size_t eval_smem() { return sizeof(MlpSmem) + EVAL_WARPS * sizeof(WarpProp); }

__global__ void __launch_bounds__(32 * EVAL_WARPS) k_dbl_eval(const SimDev *__restrict__ Sp,
                                                             const StageDev *__restrict__ stp,
                                                             const double *__restrict__ x,
                                                             const int *__restrict__ pid,
                                                             const int *__restrict__ cell,
                                                             const int *__restrict__ start,
                                                             const int *__restrict__ list,
                                                             const int *__restrict__ koff,
                                                             const int *__restrict__ comp_of,
                                                             const int *__restrict__ slot_of,
                                                             Attempt *__restrict__ att, long long sweep,
                                                             unsigned *flags, LearnedArgs la)
{
    extern __shared__ __align__(16) unsigned char smem[];
    MlpSmem &W = *reinterpret_cast<MlpSmem *>(smem);
    WarpProp *wps = reinterpret_cast<WarpProp *>(smem + sizeof(MlpSmem));
    mlp_load(W, la.w);
    __syncthreads();
    if (flags[0]) return;                          // a latched error stops the sweep (no block barrier follows)
    const SimDev &S = *Sp;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = blockIdx.x * EVAL_WARPS + warp;
    if (g >= koff[S.n_melts]) return;
    int m = 0;
    while (g >= koff[m + 1]) ++m;
    const DBC C = make_dbc(S, *stp, m, x, pid, cell, start, list, la.rec, stp->T);
    unsigned err = 0;
    Attempt a;
    learned_draw(C, ViewMap{comp_of, slot_of}, W, wps[warp], la, S.seed, sweep, g - koff[m], g, a, err);
    if (lane == 0) {
        att[g] = a;
        if (err) atomicOr(flags, err);
    }
}

// learned proposal: a stale record is re-evaluated by one warp with the
// network in shared memory; the reach of an evaluation sets the radius
struct LearnedEval {
    const SimDev *S;
    const StageDev *st;
    const double *x;
    const int *pid, *cell, *start, *list;
    const int *comp_of, *slot_of;
    long long sweep;
    unsigned *errw;              // RoundArgs::errw
    LearnedArgs la;
    const MlpSmem *W;            // set by the kernel
    WarpProp *wp;
    static constexpr int TASKS = 3;
    __device__ DBC dbc(int m) const { return make_dbc(*S, *st, m, x, pid, cell, start, list, la.rec, st->T); }
    __device__ void say(unsigned err) const
    {
        if (err && (threadIdx.x & 31) == 0) atomicOr(errw, err);
    }
    __device__ void scan(int m, int k, int g, Attempt &a)
    {
        unsigned err = 0;
        learned_draw(dbc(m), ViewMap{comp_of, slot_of}, *W, *wp, la, S->seed, sweep, k, g, a, err);
        say(err);
    }
    // probability that the partner bond proposes the swap, and that either new bond proposes the one back
    __device__ double task(int m, const Attempt &a, int t)
    {
        const DBC C = dbc(m);
        const ViewMap v{comp_of, slot_of};
        const ViewMove<ViewMap> w{v, a.kind, a.A, a.B, a.pA, a.pB, C.md.N, C.md.off};
        unsigned err = 0;
        const double p =
            t == 0 ? match_prob(C, v, *W, *wp, la, a.d, a.q, a.kind, a.A, a.B, a.pA, a.pB, err)
                   : match_prob(C, w, *W, *wp, la, t == 1 ? a.A : a.B, t == 1 ? a.pA : a.pB, a.kind, a.A, a.B, a.pA, a.pB,
                                err);
        say(err);
        return p;
    }
    __device__ bool accepts(int m, int k, const Attempt &a, const double *p) const
    {
        const double q_fwd = a.p + p[0], q_rev = p[1] + p[2];
        if (!(q_rev > 0.0) || !(q_fwd > 0.0)) {
            atomicOr(errw, ERR_DB_INTERNAL);
            return false;
        }
        return accept_u(S->seed, m, sweep, k) < exp(-a.dE / st->T) * q_rev / q_fwd;
    }
};

struct LearnedRadius {
    const unsigned long long *bmax2;
    double lim;                                    // swap bond limit (1.3)
    // cells within 2 lim + 3 max(b_max, lim) of a junction monomer, one extra
    // cell against rounding at cell faces
    __device__ int radius(const MeltDev &md) const
    {
        const double bmax = sqrt(__longlong_as_double((long long)*bmax2));
        const double reach = 2.0 * lim + 3.0 * fmax(bmax, lim);
        return (int)ceil(reach * md.invhdb) + 1;
    }
};

__global__ void __launch_bounds__(32 * EVAL_WARPS) k_dbl_rounds(RoundArgs R, LearnedEval ev)
{
    extern __shared__ __align__(16) unsigned char smem[];
    MlpSmem &W = *reinterpret_cast<MlpSmem *>(smem);
    WarpProp *wps = reinterpret_cast<WarpProp *>(smem + sizeof(MlpSmem));
    mlp_load(W, ev.la.w);
    __syncthreads();
    ev.W = &W;
    ev.wp = wps + (threadIdx.x >> 5);
    LearnedRadius pol{ev.la.bmax2, sqrt(R.sim->db_lim2)};
    rounds_body<32 * EVAL_WARPS>(ev, pol, R);
}

// longest bond of all melts, squared, as ordered binary64 bits
__global__ void __launch_bounds__(256) k_bond_max(const SimDev *__restrict__ Sp, const double *__restrict__ x,
                                                 const int *__restrict__ comp_of, unsigned long long *bmax2)
{
    const SimDev &S = *Sp;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    double r2 = 0.0;
    if (s < S.M) {
        const MeltDev &md = S.melt[melt_of(S, s)];
        const int i = (s - md.off) % md.N;
        if (i < md.N - 1) r2 = dist2_exact(x, S.Mp, md.L, md.invLf, comp_of[s], comp_of[s + 1]);
    }
    for (int o = 16; o > 0; o >>= 1) r2 = fmax(r2, __shfl_xor_sync(FULL, r2, o));
    if ((threadIdx.x & 31) == 0 && r2 > 0.0) atomicMax(bmax2, (unsigned long long)__double_as_longlong(r2));
}

// Append the sweep's log rows (attempt order, list order within an attempt) to
// the training ring: rows of attempt k go to head + off[k] (off the scan of
// the row counts), a warp copies the rows of its 32 attempts one attempt after
// the other (almost all have none).  One block walking the attempts with a
// scan of its own per 1,024 took 236 us for 80,000 attempts.
__global__ void __launch_bounds__(256) k_log_append(const int *__restrict__ logn, const int *__restrict__ off, int Ktot,
                                                   const double *__restrict__ sf, const double *__restrict__ st,
                                                   double *__restrict__ rf, double *__restrict__ rt, long long cap,
                                                   const long long *__restrict__ head, const unsigned *flags)
{
    if (flags[0]) return;
    const int k = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const int n = k < Ktot ? logn[k] : 0, o = k < Ktot ? off[k] : 0;
    // rows that an append of more than `cap` rows overwrites within itself are
    // skipped, so no two writes of one pass land on the same ring slot
    const long long base = *head, keep_from = base + off[Ktot] - cap;
    unsigned bal = __ballot_sync(FULL, n > 0);
    while (bal) {
        const int src = __ffs(bal) - 1;
        bal &= bal - 1;
        const int nn = __shfl_sync(FULL, n, src), kk = __shfl_sync(FULL, k, src);
        const long long d0 = base + __shfl_sync(FULL, o, src);
        for (int j = 0; j < nn; ++j) {
            if (d0 + j < keep_from) continue;
            const long long dst = (d0 + j) % cap;
            if (lane < 24) rf[dst * 24 + lane] = sf[((long long)kk * CAND_CAP + j) * 24 + lane];
            if (lane == 24) rt[dst] = st[(long long)kk * CAND_CAP + j];
        }
    }
}

__global__ void k_log_head(const int *__restrict__ off, int Ktot, long long *head, const unsigned *flags)
{
    if (!flags[0]) *head += off[Ktot];
}

// One bond's learned proposal in the current topology (introspection).
__global__ void __launch_bounds__(32) k_dbl_proposal(const SimDev *__restrict__ Sp, const StageDev *__restrict__ stp,
                                                    const double *__restrict__ x, const int *__restrict__ pid,
                                                    const int *__restrict__ cell, const int *__restrict__ start,
                                                    const int *__restrict__ list, const int *__restrict__ comp_of,
                                                    const int *__restrict__ slot_of, int melt, int c, int b,
                                                    LearnedArgs la, int *out_i, double *out_d, unsigned *flags)
{
    extern __shared__ __align__(16) unsigned char smem[];
    MlpSmem &W = *reinterpret_cast<MlpSmem *>(smem);
    WarpProp &wp = *reinterpret_cast<WarpProp *>(smem + sizeof(MlpSmem));
    mlp_load(W, la.w);
    __syncthreads();
    const SimDev &S = *Sp;
    const DBC C = make_dbc(S, *stp, melt, x, pid, cell, start, list, la.rec, stp->T);
    unsigned err = 0;
    // log rows of "attempt" 0 go to out_d[0 .. 48*24) (features) and out_d[48*24 ..) (targets)
    la.logf = out_d;
    la.logt = out_d + CAND_CAP * 24;
    la.logn = out_i;
    const int n = proposal(C, ViewMap{comp_of, slot_of}, W, wp, la, c, b, true, 0, err, true);
    const int lane = threadIdx.x;
    out_i[0] = n;                                  // every lane writes the same value
    for (int j = lane; j < (n > 0 ? n : 0); j += 32) {
        out_i[1 + j] = wp.cand[j].kind;
        out_i[1 + CAND_CAP + j] = wp.cand[j].d;
        out_i[1 + 2 * CAND_CAP + j] = wp.cand[j].q;
        out_d[CAND_CAP * 25 + j] = la.lambda < 1.0 ? (double)wp.s[j] : 0.0;
        out_d[CAND_CAP * 26 + j] = wp.pi[j];
    }
    if (lane == 0 && err) atomicOr(flags, err);
}

static inline int nblk(long long n, int b) { return (int)((n + b - 1) / b); }

static bool ensure_log_staging(kg_ctx *c, long long tot)
{
    if (tot <= c->log_att_cap) return true;
    dev_free(c, c->logf);
    dev_free(c, c->logt);
    dev_free(c, c->logn);
    dev_free(c, c->logoff);
    const long long cap = tot > 2 * c->log_att_cap ? tot : 2 * c->log_att_cap;
    c->logf = (double *)dev_alloc(c, sizeof(double) * 24 * CAND_CAP * (size_t)cap);
    c->logt = (double *)dev_alloc(c, sizeof(double) * CAND_CAP * (size_t)cap);
    c->logn = (int *)dev_alloc(c, sizeof(int) * (size_t)cap);
    // offsets of the attempts' rows, and the block sums of their scan
    c->logoff = (int *)dev_alloc(c, sizeof(int) * ((size_t)cap + 1 + (size_t)cap / 1024 + 2));
    c->log_att_cap = (c->logf && c->logt && c->logn && c->logoff) ? cap : 0;
    return c->log_att_cap > 0;
}

static LearnedArgs make_args(kg_ctx *c, double lambda, bool log)
{
    LearnedArgs la;
    la.lambda = lambda;
    la.w = (const MlpSmem *)c->mlp_blob;
    la.logf = log ? c->logf : nullptr;
    la.logt = log ? c->logt : nullptr;
    la.logn = log ? c->logn : nullptr;
    la.bmax2 = c->bmax2;
    la.rec = c->dbrec;
    return la;
}

cudaError_t db_sweep_learned(kg_ctx *c, const std::vector<long long> &K, double lambda, long long *host_stats)
{
    cudaStream_t st = c->stream;
    const int nm = c->sim.n_melts;
    long long tot = 0;
    for (long long k : K) tot += k;
    const bool log = c->train_cap > 0 && ensure_log_staging(c, tot > 0 ? tot : 1);
    const LearnedArgs la = make_args(c, lambda, log);
    db_bin(c, K);
    cudaMemsetAsync(c->bmax2, 0, sizeof(unsigned long long), st);
    k_bond_max<<<nblk(c->M, 256), 256, 0, st>>>(c->d_sim, c->x, c->comp_of, c->bmax2);
    Attempt *att = (Attempt *)c->att;
    if (tot > 0) {
        cudaFuncSetAttribute(k_dbl_eval, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)eval_smem());
        k_dbl_eval<<<nblk(tot, EVAL_WARPS), 32 * EVAL_WARPS, eval_smem(), st>>>(
            c->d_sim, c->d_stage, c->x, c->pid, c->dbcell, c->dbstart, c->dblist, c->koff, c->comp_of, c->slot_of,
            att, c->sweep, c->flags, la);
    }
    // ordered commit in rounds (kg_db.cuh)
    db_rounds_reset(c);
    cudaFuncSetAttribute(k_dbl_rounds, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)eval_smem());
    const RoundArgs ra = round_args(c);
    const LearnedEval ev{c->d_sim, c->d_stage, c->x, c->pid, c->dbcell, c->dbstart, c->dblist,
                         c->comp_of, c->slot_of, c->sweep, ra.errw, la, nullptr, nullptr};
    const cudaError_t e = rounds_launch(c, k_dbl_rounds, 32 * EVAL_WARPS, eval_smem(), tot, nm, ra, ev);
    if (e != cudaSuccess) return e;
    c->launches += 2;
    if (log && tot > 0) {
        scan_counts(c, c->logn, c->logoff, (int)tot, c->logoff + tot + 1);
        k_log_append<<<nblk(tot, 256), 256, 0, st>>>(c->logn, c->logoff, (int)tot, c->logf, c->logt, c->trainf,
                                                     c->traint, c->train_cap, c->d_train_head, c->flags);
        k_log_head<<<1, 1, 0, st>>>(c->logoff, (int)tot, c->d_train_head, c->flags);
        c->launches += 3;
        ++c->launches;
    }
    db_finish(c, host_stats);
    return cudaSuccess;
}

bool db_proposal(kg_ctx *c, int melt, int chain, int bond, double lambda, int *h_n, int *h_ints, double *h_f,
                 double *h_s, double *h_pi)
{
    cudaStream_t st = c->stream;
    std::vector<long long> K(c->sim.n_melts, 0);
    db_bin(c, K);
    const size_t nd = CAND_CAP * 27, ni = 1 + 3 * CAND_CAP;
    double *dd = (double *)dev_alloc(c, sizeof(double) * nd);
    int *di = (int *)dev_alloc(c, sizeof(int) * ni);
    if (!dd || !di) {
        dev_free(c, dd);
        dev_free(c, di);
        return false;
    }
    const LearnedArgs la = make_args(c, lambda, false);
    const size_t sm = sizeof(MlpSmem) + sizeof(WarpProp);
    cudaFuncSetAttribute(k_dbl_proposal, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    k_dbl_proposal<<<1, 32, sm, st>>>(c->d_sim, c->d_stage, c->x, c->pid, c->dbcell, c->dbstart, c->dblist,
                                      c->comp_of, c->slot_of, melt, chain, bond, la, di, dd, c->flags);
    ++c->launches;
    std::vector<double> hd(nd);
    std::vector<int> hi(ni);
    cudaMemcpyAsync(hd.data(), dd, sizeof(double) * nd, cudaMemcpyDeviceToHost, st);
    cudaMemcpyAsync(hi.data(), di, sizeof(int) * ni, cudaMemcpyDeviceToHost, st);
    const bool ok = cudaStreamSynchronize(st) == cudaSuccess;
    dev_free(c, dd);
    dev_free(c, di);
    if (!ok) return false;
    const int n = hi[0];
    *h_n = n;
    for (int j = 0; j < (n > 0 ? n : 0); ++j) {
        h_ints[j] = hi[1 + j];
        h_ints[CAND_CAP + j] = hi[1 + CAND_CAP + j];
        h_ints[2 * CAND_CAP + j] = hi[1 + 2 * CAND_CAP + j];
        for (int i = 0; i < 24; ++i) h_f[j * 24 + i] = hd[j * 24 + i];
        h_s[j] = hd[CAND_CAP * 25 + j];
        h_pi[j] = hd[CAND_CAP * 26 + j];
    }
    return true;
}

}  // namespace kg
