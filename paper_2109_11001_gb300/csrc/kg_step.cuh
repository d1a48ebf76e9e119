// kg_step.cuh -- arithmetic of the mixed path's MD step, shared by the one-step
// kernel (kg_step.cu) and the resident kernels (kg_resident*.cu): all give the
// same bits.
#pragma once
#include <cuda_runtime.h>

#include "kg_host.h"
#include "kg_rebuild.cuh"

namespace kg {

struct MeltStep {
    int off, nc;
    float h, L, invL, kappa;
};

struct StepArgs {
    const float4 *recb;      // build records: offset from the Verlet-cell corner, packed cell coordinates
    const float4 *dcur;      // displacement since the build (this step)
    float4 *dnext;           //   ... after this step
    const float4 *pcur;      // gather records recb + dcur
    float4 *pnext;           //   ... after this step
    float *u;                // [3][Mp] velocities v_{n-1/2}
    const unsigned *nl;      // Verlet list, column-major [maxnb][Mp], entries j | q << IDX_BITS
    const int *nn;           // list lengths
    const int *slot_of;      // compute index -> chain-major slot (keys the noise)
    const int4 *bp;          // compute indices of chain partners s-2, s-1, s+1, s+2 (-1 past an end)
    unsigned *flags;         // [0] error bits, [1] rebuild request
    const long long *stepp;  // index of the step being run (in a loop: of the last one before the pass)
    LoopDev *loop;           // captured step loop (null: none), and the step's place in its body
    int k;
    unsigned long long seed;
    int M, Mp, n_melts;
    float rc2, half_skin2;
    float dt, gamma, amp;    // Langevin: u += dt (F - gamma u + amp g), amp = sqrt(2 gamma T / dt)
    float c1xn, c2x6, nf;    // fr = (6 c2 r^-6 - n c1 r^-n) / r^2  (U = c1 r^-n - c2 r^-6 + 1)
    float kf, R0sq, inv_R0sq, qmin, kf_qmin, four_R0sq;   // FENE k_n, R0^2, continuation beyond r*
    MeltStep melt[MAX_MELTS];
};

// r^-n from r^2, 1/r^2 and 1/r^6; N4 = 4n (0: any other n, from exp2/log2)
template <int N4>
__device__ __forceinline__ float inv_rn(float r2, float ir2, float ir6, float nf)
{
    if constexpr (N4 == 0) {
        return exp2f(-0.5f * nf * log2f(r2));
    } else if constexpr (N4 == 23) {                 // n = 23/4: r^-6 r^(1/4)
        return ir6 * sqrtf(sqrtf(sqrtf(r2)));
    } else if constexpr (N4 == 26) {                 // n = 13/2: r^-6 r^(-1/2)
        return ir6 * sqrtf(rsqrtf(r2));
    } else {
        static_assert(N4 % 4 == 0, "integer n");
        constexpr int n = N4 / 4;
        float p;
        if constexpr (n >= 6) {
            p = ir6;
#pragma unroll
            for (int k = 3; k < n / 2; ++k) p *= ir2;
        } else {
            p = ir2;
#pragma unroll
            for (int k = 1; k < n / 2; ++k) p *= ir2;
        }
        if constexpr (n & 1) p *= rsqrtf(r2);
        return p;
    }
}

// (dU_MLJ^n/dr) / r at r^2 (binary32)
template <int N4>
__device__ __forceinline__ float mlj_fr32(const StepArgs &P, float r2)
{
    const float ir2 = __fdividef(1.0f, r2);
    const float ir6 = ir2 * ir2 * ir2;
    const float rn = inv_rn<N4>(r2, ir2, ir6, P.nf);
    return __fmul_rn(fmaf(P.c2x6, ir6, -__fmul_rn(P.c1xn, rn)), ir2);
}

__device__ __forceinline__ int melt_index(const StepArgs &P, int slot)
{
    int m = 0;
    while (m + 1 < P.n_melts && slot >= P.melt[m + 1].off) ++m;
    return m;
}

// Arithmetic of the step written with explicit roundings: a sum of two
// products leaves the compiler a choice of which one to fuse, and the choice
// can differ between the kernels that inline the step (standalone and
// persistent), which must give the same bits.  fmaf is always fused,
// __fmul_rn / __fadd_rn / __fsub_rn never.
__device__ __forceinline__ float dot3(float3 a, float3 b)
{
    return fmaf(a.z, b.z, fmaf(a.y, b.y, __fmul_rn(a.x, b.x)));
}

__device__ __forceinline__ void axpy3(float a, float3 x, float3 &y)   // y += a x
{
    y.x = fmaf(a, x.x, y.x);
    y.y = fmaf(a, x.y, y.y);
    y.z = fmaf(a, x.z, y.z);
}

__device__ __forceinline__ float3 sub3(float3 a, float3 b)
{
    return make_float3(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y), __fsub_rn(a.z, b.z));
}

// a inv - c b: one term of the gradient of cos theta
__device__ __forceinline__ float3 bend_g(float3 a, float inv, float c, float3 b)
{
    return make_float3(fmaf(-c, b.x, __fmul_rn(a.x, inv)), fmaf(-c, b.y, __fmul_rn(a.y, inv)),
                       fmaf(-c, b.z, __fmul_rn(a.z, inv)));
}

// Bond (Eq. 10) and bending (Eq. 4) forces on the monomer whose gather
// record is pi, from its chain partners bp = (s-2, s-1, s+1, s+2);
// rec(k, j): the gather record of partner k (0..3), compute index j; add(k, a,
// x): term k of the force, F += a x, called in the order k = 0 ... 4 (two
// bonds, three angles) for the terms that exist.
template <int N4, class REC, class ADD>
__device__ __forceinline__ void bonded32(const StepArgs &P, REC rec, ADD add, const MeltStep &md, float4 pi, int4 bp,
                                         unsigned &err)
{
    const bool hm2 = bp.x >= 0, hm1 = bp.y >= 0, hp1 = bp.z >= 0, hp2 = bp.w >= 0;
    float3 rm2 = make_float3(0.f, 0.f, 0.f), rm1 = rm2, rp1 = rm2, rp2 = rm2;
    if (hm1) rm1 = rec_rel(pi, rec(1, bp.y), md.nc, md.h, md.L, md.invL);
    if (hm2) rm2 = rec_rel(pi, rec(0, bp.x), md.nc, md.h, md.L, md.invL);
    if (hp1) rp1 = rec_rel(pi, rec(2, bp.z), md.nc, md.h, md.L, md.invL);
    if (hp2) rp2 = rec_rel(pi, rec(3, bp.w), md.nc, md.h, md.L, md.invL);
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        if (side == 0 ? hm1 : hp1) {
            const float3 d = side == 0 ? rm1 : rp1;
            const float r2 = dot3(d, d);
            float q = 1.0f - r2 * P.inv_R0sq, fr;
            if (P.qmin > 0.0f && q < P.qmin) {          // continuation beyond r* (kg_params.fene_qmin)
                fr = P.kf_qmin;
                if (!(r2 < P.four_R0sq)) err |= ERR_OVERSTRETCH;
            } else {
                if (!(r2 < P.R0sq)) err |= ERR_OVERSTRETCH;
                q = fmaxf(q, 1e-6f);                    // finite even when flagged
                fr = P.kf * __fdividef(1.0f, q);
            }
            const float fl = mlj_fr32<N4>(P, r2);
            fr += r2 < P.rc2 ? fl : 0.0f;
            add(side, fr, d);
        }
    }
    const float kap = md.kappa;
    if (kap != 0.0f) {
        const float3 Bm2 = sub3(rm1, rm2);
        const float3 Bm1 = make_float3(-rm1.x, -rm1.y, -rm1.z), B0 = rp1;
        const float3 Bp1 = sub3(rp2, rp1);
        if (hm1 && hp1) {                     // vertex s: force kappa (g1 - g2)
            const float l1 = dot3(Bm1, Bm1), l2 = dot3(B0, B0);
            const float inv = rsqrtf(__fmul_rn(l1, l2)), cs = __fmul_rn(dot3(Bm1, B0), inv);
            const float c1 = __fmul_rn(cs, __fdividef(1.0f, l1)), c2 = __fmul_rn(cs, __fdividef(1.0f, l2));
            add(2, kap, sub3(bend_g(B0, inv, c1, Bm1), bend_g(Bm1, inv, c2, B0)));
        }
        if (hp2) {                            // vertex s+1, s its first end: -kappa g1
            const float l1 = dot3(B0, B0), l2 = dot3(Bp1, Bp1);
            const float inv = rsqrtf(__fmul_rn(l1, l2)), cs = __fmul_rn(dot3(B0, Bp1), inv);
            const float c1 = __fmul_rn(cs, __fdividef(1.0f, l1));
            add(3, -kap, bend_g(Bp1, inv, c1, B0));
        }
        if (hm2) {                            // vertex s-1, s its last end: +kappa g2
            const float l1 = dot3(Bm2, Bm2), l2 = dot3(Bm1, Bm1);
            const float inv = rsqrtf(__fmul_rn(l1, l2)), cs = __fmul_rn(dot3(Bm2, Bm1), inv);
            const float c2 = __fmul_rn(cs, __fdividef(1.0f, l2));
            add(4, kap, bend_g(Bm2, inv, c2, Bm1));
        }
    }
}

// the stencil offsets of the 27 codes, one word table per axis (96 floats of shared memory)
__device__ __forceinline__ void step_block_setup(float *dk)
{
    if (threadIdx.x < 27) {
        const int q = threadIdx.x;
        dk[q] = (float)(q % 3 - 1);
        dk[32 + q] = (float)((q / 3) % 3 - 1);
        dk[64 + q] = (float)(q / 9 - 1);
    }
}

constexpr int STEP_ILP = 4;      // Verlet-list entries in flight per lane
// One tile of blockDim threads (all threads of the block call it together):
// the step of the monomers of threads t0 + threadIdx.x.  TPM threads per
// monomer (1 or 2, adjacent lanes): the lanes split the list (entries k =
// sub, sub + TPM, ...); with two, lane 0 adds the bonded terms and lane 1
// draws the noise, the forces are combined with a shuffle, and lane 0 writes
// the state.  The pair loop comes first and holds only its own state (the
// own gather record, the force, the entries in flight), so the kernel fits
// 32 registers at full occupancy; the bonded terms, the noise and the build
// record and displacement for the update follow.  The pair loop runs to the
// warp's longest list in groups of STEP_ILP entries with per-lane
// predicates: an entry past the lane's own list becomes the lane's own record
// with the zero shift (code 13), a valid gather whose term is masked.
// READ_ONLY: nothing it loads is written in the same launch (non-coherent
// loads).  vote(rebuild, err), by every lane of the warp: its monomer left its
// skin, and its error bits.  go(), by every thread once its first loads are
// under way: false if the block does not run the step after all.
template <bool READ_ONLY, typename T>
__device__ __forceinline__ T step_ld(const T *p)
{
    if constexpr (READ_ONLY) return __ldg(p);
    else return *p;
}

template <int N4, int TPM, bool READ_ONLY, class VOTE, class GO>
__device__ __forceinline__ void step_tile(const StepArgs &P, int t0, const float4 *dcur, float4 *dnext,
                                          const float4 *pcur, float4 *pnext, long long step, const float *dk,
                                          VOTE vote, GO go)
{
    constexpr bool RO = READ_ONLY;
    const int lane = threadIdx.x & 31;
    const int t = t0 + threadIdx.x;
    const int s = t / TPM, sub = t % TPM;
    const bool live = s < P.M;
    const int cnt = live ? step_ld<RO>(P.nn + s) : 0;
    unsigned err = 0;
    float3 F = make_float3(0.f, 0.f, 0.f), gn = F;
    int slot = 0;
    float4 pi = make_float4(0.f, 0.f, 0.f, 0.f);
    if (live) {
        slot = __ldg(P.slot_of + s);
        pi = step_ld<RO>(pcur + s);
    }
    if (!go()) return;                     // the same for the whole block
    const int kmax = __reduce_max_sync(0xffffffffu, cnt);
    const int m = live ? melt_index(P, slot) : 0;
    const MeltStep &md = P.melt[m];
    const float h = md.h, rc2 = P.rc2;
    const unsigned self = (unsigned)(live ? s : 0) | (13u << IDX_BITS);
    const size_t Mp = (size_t)P.Mp;
    const unsigned *col = P.nl + (live ? s : 0);
    for (int k0 = sub; k0 < kmax; k0 += STEP_ILP * TPM) {
        unsigned e[STEP_ILP];
        float4 pj[STEP_ILP];
#pragma unroll
        for (int i = 0; i < STEP_ILP; ++i) {
            const int k = k0 + i * TPM;
            e[i] = k < cnt ? step_ld<RO>(col + (size_t)k * Mp) : self;
        }
#pragma unroll
        for (int i = 0; i < STEP_ILP; ++i) pj[i] = step_ld<RO>(pcur + (e[i] & IDX_MASK));
#pragma unroll
        for (int i = 0; i < STEP_ILP; ++i) {
            const unsigned q = e[i] >> IDX_BITS;
            const float dx = fmaf(dk[q], h, pj[i].x - pi.x);
            const float dy = fmaf(dk[32 + q], h, pj[i].y - pi.y);
            const float dz = fmaf(dk[64 + q], h, pj[i].z - pi.z);
            const float r2 = fmaf(dz, dz, fmaf(dy, dy, __fmul_rn(dx, dx)));
            float fr = mlj_fr32<N4>(P, r2);
            fr = (k0 + i * TPM < cnt && r2 < rc2) ? fr : 0.0f;
            F.x = fmaf(fr, dx, F.x); F.y = fmaf(fr, dy, F.y); F.z = fmaf(fr, dz, F.z);
        }
    }
    float4 rb = make_float4(0.f, 0.f, 0.f, 0.f), dc = rb;
    if (live) {
        if (sub == 0) bonded32<N4>(P, [&](int, int j) { return step_ld<RO>(pcur + j); },
                                   [&](int, float a, float3 x) { axpy3(a, x, F); }, md, pi, __ldg(P.bp + s), err);
        if (sub == TPM - 1)
            gn = gauss3_f(draw(P.seed, m, 0, (unsigned long long)step, (uint32_t)(slot - md.off)));
        rb = step_ld<RO>(P.recb + s);
        dc = step_ld<RO>(dcur + s);
    }
    if (TPM == 2) {                        // every lane takes part: s is shared by lanes 2i, 2i+1
        F.x += __shfl_xor_sync(0xffffffffu, F.x, 1);
        F.y += __shfl_xor_sync(0xffffffffu, F.y, 1);
        F.z += __shfl_xor_sync(0xffffffffu, F.z, 1);
        const int src = lane | 1;
        gn.x = __shfl_sync(0xffffffffu, gn.x, src);
        gn.y = __shfl_sync(0xffffffffu, gn.y, src);
        gn.z = __shfl_sync(0xffffffffu, gn.z, src);
    }
    bool rebuild = false;
    if (live && sub == 0) {
        const int Mpi = P.Mp;
        float *u = P.u;
        float3 v = make_float3(u[s], u[Mpi + s], u[2 * Mpi + s]);
        v.x = fmaf(P.dt, fmaf(P.amp, gn.x, fmaf(-P.gamma, v.x, F.x)), v.x);
        v.y = fmaf(P.dt, fmaf(P.amp, gn.y, fmaf(-P.gamma, v.y, F.y)), v.y);
        v.z = fmaf(P.dt, fmaf(P.amp, gn.z, fmaf(-P.gamma, v.z, F.z)), v.z);
        u[s] = v.x; u[Mpi + s] = v.y; u[2 * Mpi + s] = v.z;
        float4 d = dc;
        d.x = fmaf(P.dt, v.x, d.x); d.y = fmaf(P.dt, v.y, d.y); d.z = fmaf(P.dt, v.z, d.z);
        dnext[s] = d;
        pnext[s] = make_float4(rb.x + d.x, rb.y + d.y, rb.z + d.z, rb.w);
        rebuild = fmaf(d.z, d.z, fmaf(d.y, d.y, __fmul_rn(d.x, d.x))) > P.half_skin2;
        if (!isfinite(v.x + v.y + v.z)) err |= ERR_NONFINITE;
    }
    vote(rebuild, err);
}

// 4n of a stage exponent with its own kernel instantiation, 0 otherwise
int n4_of(double n);
// the by-value arguments of a step from gather buffer cur (kg_step.cu)
StepArgs step_args(const kg_ctx *c, int cur);
NlArgs nl_args(const kg_ctx *c);                 // kg_md.cu

}  // namespace kg
