// kg_md.cu -- molecular-dynamics kernels of the GB300 DBH library.
//
//  * cell binning + counting sort + Verlet-list build (every rebuild);
//  * one fused kernel per MD step: U_MLJ^n pairs over the Verlet list (Eq. 6),
//    U_bond^n bonds (Eq. 10), kappa (1 - cos theta) bending (Eq. 4), Langevin
//    friction and Philox noise, and the leapfrog update of (x, u);
//  * a force/energy kernel for observables and parity checks.
// Thread per monomer in compute order: the per-monomer arrays are kept sorted
// by Verlet-list cell (re-sorted every few hundred steps), so a warp's
// neighbours sit in a few contiguous runs of memory.  bp[i] holds the compute
// indices of the monomers two and one before and after along the chain
// (-1 past a chain end); slot_of[i] is the chain-major slot c*N + i, which keys
// the random draws so results do not depend on the order.
#include <cuda_runtime.h>

#include <algorithm>

#include "kg_host.h"
#include "kg_rebuild.cuh"

namespace kg {

// ---------------------------------------------------------------------------
// pair and bond terms (binary32 and binary64 forms of the same formulas)
// U_MLJ^n(r) = c1 r^-n - c2 r^-6 + 1 for r < r_c (Eqs. 5-6, shifted by +epsilon);
// fr = (dU/dr)/r, so the force on i from j at d = x_j - x_i is fr * d.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float mlj_fr(const StageDev &st, float r2, float &U)
{
    const float ir2 = __fdividef(1.0f, r2);
    const float ir6 = ir2 * ir2 * ir2;
    float rn;
    if (st.nint == 12) {                 // WCA (Eq. 2): the production potential
        rn = ir6 * ir6;
    } else if (st.nkind == 1) {
        float p = 1.0f;
        for (int k = 0; k < (st.nint >> 1); ++k) p *= ir2;
        if (st.nint & 1) p *= rsqrtf(r2);
        rn = p;
    } else if (st.nkind == 2) {          // n = 23/4: r^-6 r^(1/4)
        rn = ir6 * sqrtf(sqrtf(sqrtf(r2)));
    } else if (st.nkind == 3) {          // n = 13/2: r^-6 r^(-1/2)
        rn = ir6 * sqrtf(rsqrtf(r2));
    } else {
        rn = exp2f(-0.5f * st.nf * log2f(r2));
    }
    U = st.c1f * rn - st.c2f * ir6 + 1.0f;
    return (st.c2x6f * ir6 - st.c1xnf * rn) * ir2;
}

__device__ __forceinline__ double mlj_fr(const StageDev &st, double r2, double &U)
{
    const double ir2 = 1.0 / r2;
    const double ir6 = ir2 * ir2 * ir2;
    double rn;
    if (st.nkind == 1) {
        double p = 1.0;
        for (int k = 0; k < (st.nint >> 1); ++k) p *= ir2;
        if (st.nint & 1) p *= rsqrt(r2);
        rn = p;
    } else if (st.nkind == 2) {
        rn = ir6 * sqrt(sqrt(sqrt(r2)));
    } else if (st.nkind == 3) {
        rn = ir6 * sqrt(rsqrt(r2));
    } else {
        rn = exp2(-0.5 * st.n * log2(r2));
    }
    U = st.c1 * rn - st.c2 * ir6 + 1.0;
    return (6.0 * st.c2 * ir6 - st.n * st.c1 * rn) * ir2;
}

template <typename T> struct V3;
template <> struct V3<float> { using t = float3; };
template <> struct V3<double> { using t = double3; };

template <typename T> __device__ __forceinline__ typename V3<T>::t mk(T a, T b, T c);
template <> __device__ __forceinline__ float3 mk<float>(float a, float b, float c) { return make_float3(a, b, c); }
template <> __device__ __forceinline__ double3 mk<double>(double a, double b, double c) { return make_double3(a, b, c); }

template <typename T3> __device__ __forceinline__ auto dot3(T3 a, T3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
template <typename T3> __device__ __forceinline__ T3 sub3(T3 a, T3 b) { return T3{a.x - b.x, a.y - b.y, a.z - b.z}; }

template <typename T> __device__ __forceinline__ T st_c(const StageDev &st, int which);
template <> __device__ __forceinline__ float st_c<float>(const StageDev &st, int w)
{
    return w == 0 ? st.kfenef : w == 1 ? st.R0sqf : w == 2 ? st.dtf : w == 3 ? st.gammaf : w == 4 ? st.ampf
         : w == 5 ? st.qminf : w == 6 ? st.r2starf : st.ustarf;
}
template <> __device__ __forceinline__ double st_c<double>(const StageDev &st, int w)
{
    return w == 0 ? st.kfene : w == 1 ? st.R0sq : w == 2 ? st.dt : w == 3 ? st.gamma : w == 4 ? st.amp
         : w == 5 ? st.qmin : w == 6 ? st.r2star : st.ustar;
}

__device__ __forceinline__ float flog(float a) { return logf(a); }
__device__ __forceinline__ double flog(double a) { return log(a); }
__device__ __forceinline__ float frsqrt(float a) { return rsqrtf(a); }
__device__ __forceinline__ double frsqrt(double a) { return rsqrt(a); }
__device__ __forceinline__ float frcp(float a) { return __fdividef(1.0f, a); }
__device__ __forceinline__ double frcp(double a) { return 1.0 / a; }

// ---------------------------------------------------------------------------
// position access policies
// ---------------------------------------------------------------------------
// binary32 gather records p = offset from the build-time cell corner +
// displacement since the build (w: packed cell coordinates).  A Verlet-list
// entry carries the image shift of its pair (the stencil code), so a listed
// pair costs one gather and one table lookup; chain partners, which are not
// in the list, take the shift from the cell codes.
struct GeoMixed {
    using T = float;
    using T3 = float3;
    const float4 *__restrict__ pg;
    const float4 *__restrict__ shtab;    // SHIFT_SLOTS shift vectors per melt
    const float4 *__restrict__ sht;
    int nc;
    float h, L, invL;
    float4 pi;
    __device__ __forceinline__ void melt(const MeltDev &md, int m)
    {
        nc = md.nc; h = md.hf; L = md.Lf; invL = md.invLf;
        sht = shtab + SHIFT_SLOTS * m;
    }
    __device__ __forceinline__ void self(int s) { pi = __ldg(pg + s); }
    __device__ __forceinline__ float3 rel_nl(unsigned e) const
    {
        const float4 pj = __ldg(pg + (e & IDX_MASK));
        const float4 sh = __ldg(sht + (e >> IDX_BITS));
        return make_float3((pj.x - pi.x) + sh.x, (pj.y - pi.y) + sh.y, (pj.z - pi.z) + sh.z);
    }
    __device__ __forceinline__ float3 rel(int j) const { return rec_rel(pi, __ldg(pg + j), nc, h, L, invL); }
};

struct GeoF64 {
    using T = double;
    using T3 = double3;
    const double4_32a *__restrict__ pos;
    double L, invL;
    double4_32a pi;
    __device__ __forceinline__ void melt(const MeltDev &md, int) { L = md.L; invL = md.invL; }
    __device__ __forceinline__ void self(int s) { pi = pos[s]; }
    __device__ __forceinline__ double3 rel(int j) const
    {
        const double4_32a pj = pos[j];
        double dx = pj.x - pi.x, dy = pj.y - pi.y, dz = pj.z - pi.z;
        dx -= L * rint(dx * invL);
        dy -= L * rint(dy * invL);
        dz -= L * rint(dz * invL);
        return make_double3(dx, dy, dz);
    }
    __device__ __forceinline__ double3 rel_nl(unsigned e) const { return rel((int)(e & IDX_MASK)); }
};

template <typename T, typename T3>
__device__ __forceinline__ void pair_term(const StageDev &st, T rc2, T3 d, T3 &F, double *e)
{
    const T r2 = dot3(d, d);
    if (r2 < rc2) {
        T U;
        const T fr = mlj_fr(st, r2, U);
        F.x += fr * d.x; F.y += fr * d.y; F.z += fr * d.z;
        e[0] += 0.5 * (double)U;
        e[3] -= 0.5 * (double)(fr * r2);
    }
}

// Pair forces on s from its Verlet list (both directions are stored), four
// entries in flight.
template <class G>
__device__ __forceinline__ void pair_forces(const G &g, const SimDev &S, const StageDev &st, int s,
                                            const unsigned *__restrict__ nl, int cnt,
                                            typename G::T3 &F, double *e)
{
    using T = typename G::T;
    using T3 = typename G::T3;
    const T rc2 = (T)S.rc2;
    const size_t step = (size_t)S.Mp;
    const unsigned *__restrict__ col = nl + s;
    int k = 0;
    for (; k + 3 < cnt; k += 4, col += 4 * step) {
        const unsigned e0 = __ldg(col), e1 = __ldg(col + step);
        const unsigned e2 = __ldg(col + 2 * step), e3 = __ldg(col + 3 * step);
        const T3 d0 = g.rel_nl(e0), d1 = g.rel_nl(e1), d2 = g.rel_nl(e2), d3 = g.rel_nl(e3);
        pair_term(st, rc2, d0, F, e);
        pair_term(st, rc2, d1, F, e);
        pair_term(st, rc2, d2, F, e);
        pair_term(st, rc2, d3, F, e);
    }
    for (; k < cnt; ++k, col += step) pair_term(st, rc2, g.rel_nl(__ldg(col)), F, e);
}

// Bond (Eq. 10) and bending (Eq. 4) forces on s from its chain partners.
template <class G>
__device__ __forceinline__ void bonded_forces(const G &g, const StageDev &st, const MeltDev &md,
                                              typename G::T rc2, int4 bp, typename G::T3 &F, double *e,
                                              unsigned &err)
{
    using T = typename G::T;
    using T3 = typename G::T3;
    // chain neighbours: bp = (s-2, s-1, s+1, s+2) along the chain, -1 past an end
    const bool hm2 = bp.x >= 0, hm1 = bp.y >= 0, hp1 = bp.z >= 0, hp2 = bp.w >= 0;
    T3 rm2 = mk<T>(0, 0, 0), rm1 = mk<T>(0, 0, 0), rp1 = mk<T>(0, 0, 0), rp2 = mk<T>(0, 0, 0);
    if (hm1) rm1 = g.rel(bp.y);
    if (hm2) rm2 = g.rel(bp.x);
    if (hp1) rp1 = g.rel(bp.z);
    if (hp2) rp2 = g.rel(bp.w);
    // bonds: U_MLJ^n + FENE(k_n) (Eq. 10)
    const T kf = st_c<T>(st, 0), R0sq = st_c<T>(st, 1);
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        if ((side == 0 && hm1) || (side == 1 && hp1)) {
            const T3 d = side == 0 ? rm1 : rp1;
            const T r2 = dot3(d, d);
            const T qmin = st_c<T>(st, 5);
            T q = (T)1 - r2 / R0sq, fr, Uf = 0;
            if (qmin > (T)0 && q < qmin) {           // continuation beyond r* (kg_params.fene_qmin)
                fr = kf * frcp(qmin);
                if (!(r2 < (T)4 * R0sq)) err |= ERR_OVERSTRETCH;
                Uf = st_c<T>(st, 7) + kf * (r2 - st_c<T>(st, 6)) / ((T)2 * qmin);
            } else {
                if (!(r2 < R0sq)) err |= ERR_OVERSTRETCH;
                q = fmax(q, (T)1e-6);                    // finite even when flagged
                fr = kf * frcp(q);
                Uf = (T)-0.5 * kf * R0sq * flog(q);
            }
            T U = 0;
            if (r2 < rc2) fr += mlj_fr(st, r2, U);
            F.x += fr * d.x; F.y += fr * d.y; F.z += fr * d.z;
            e[1] += 0.5 * ((double)U + (double)Uf);
            e[3] -= 0.5 * (double)(fr * r2);
        }
    }
    // bending kappa (1 - b1.b2 / |b1||b2|) at the vertices s-1, s, s+1
    const T kap = (T)md.kappa;
    if (kap != (T)0) {
        const T3 Bm2 = sub3(rm1, rm2), Bm1 = mk<T>(-rm1.x, -rm1.y, -rm1.z), B0 = rp1, Bp1 = sub3(rp2, rp1);
        if (hm1 && hp1) {                    // vertex s: force kappa (g1 - g2)
            const T l1 = dot3(Bm1, Bm1), l2 = dot3(B0, B0), inv = frsqrt(l1 * l2), cs = dot3(Bm1, B0) * inv;
            const T c1 = cs * frcp(l1), c2 = cs * frcp(l2);
            F.x += kap * ((B0.x * inv - c1 * Bm1.x) - (Bm1.x * inv - c2 * B0.x));
            F.y += kap * ((B0.y * inv - c1 * Bm1.y) - (Bm1.y * inv - c2 * B0.y));
            F.z += kap * ((B0.z * inv - c1 * Bm1.z) - (Bm1.z * inv - c2 * B0.z));
            e[2] += (double)kap * (1.0 - (double)cs);
        }
        if (hp2) {                           // vertex s+1, s is its first end: -kappa g1
            const T l1 = dot3(B0, B0), l2 = dot3(Bp1, Bp1), inv = frsqrt(l1 * l2), cs = dot3(B0, Bp1) * inv;
            const T c1 = cs * frcp(l1);
            F.x -= kap * (Bp1.x * inv - c1 * B0.x);
            F.y -= kap * (Bp1.y * inv - c1 * B0.y);
            F.z -= kap * (Bp1.z * inv - c1 * B0.z);
        }
        if (hm2) {                           // vertex s-1, s is its last end: +kappa g2
            const T l1 = dot3(Bm2, Bm2), l2 = dot3(Bm1, Bm1), inv = frsqrt(l1 * l2), cs = dot3(Bm2, Bm1) * inv;
            const T c2 = cs * frcp(l2);
            F.x += kap * (Bm2.x * inv - c2 * Bm1.x);
            F.y += kap * (Bm2.y * inv - c2 * Bm1.y);
            F.z += kap * (Bm2.z * inv - c2 * Bm1.z);
        }
    }
}

// Conservative force on slot s (chain position i of N) and its
// shares of the energies: e[0] pair (1/2 per pair), e[1] bond (1/2 per bond),
// e[2] bending (the angle whose vertex is s), e[3] virial (1/2 per pair/bond).
template <class G>
__device__ __forceinline__ typename G::T3 force_on(const G &g, const SimDev &S, const StageDev &st,
                                                   const MeltDev &md, int s, int4 bp,
                                                   const unsigned *__restrict__ nl, int cnt,
                                                   double *e, unsigned &err)
{
    using T = typename G::T;
    typename G::T3 F = mk<T>(0, 0, 0);
    pair_forces(g, S, st, s, nl, cnt, F, e);
    bonded_forces(g, st, md, (T)S.rc2, bp, F, e, err);
    return F;
}

// ---------------------------------------------------------------------------
// fused MD step, binary64 path: forces at x_n, then u <- u + dt F_n,
// x <- x + dt u with F_n = F_c - gamma u + sqrt(2 gamma T / dt) g_n,
// g_n = Philox normals (the mixed path's step kernel is in kg_step.cu)
//
// The binary64 pipe (two lanes a clock on an SM) bounds it, so what need not
// go there does not:
//  * a list entry is first looked at in binary32, on the same gather records as
//    the mixed path (offset from the build-time cell corner + displacement, a
//    shift for the stencil code), with a margin above their rounding; only the
//    pairs that may lie within r_c, about a third to a half of the list, take
//    the binary64 minimum image, distance and force;
//  * the near pairs of a warp's 32 monomers form one queue, worked through a pair
//    a lane; the results go through shared memory to their owners, who add them
//    in list order.  Popping its own pairs, a lane waited for the largest of 32
//    numbers of near pairs (about 9 against a mean of 4 to 5);
//  * a bond's inverse length is one reciprocal square root that serves its own
//    1/r^2, both its angles and all their gradients, each corrected by a Newton
//    step: without it (and with r^-12 as a square) a step's forces were twice as
//    far from 128 bits (3.0e-14 of a force against 1.42e-14 of plain divides and
//    square roots; with it 1.42e-14).
// Blocks of 64, whatever block_size says: the pipe is the SM's, so the SM with
// the most blocks sets the time, and 80,000 monomers are 4.1 blocks of 128 per
// SM (five on some) but 8.2 of 64.  80,000 monomers, n = 12, skin 0.3, 50 steps
// with 14 list builds: 9016 -> 5290 us (4990 without the corrections; at
// exponents that take log2 and exp2 a pair is four times the work).  200,000, n =
// 2: 17170 -> 10900 us.
// ---------------------------------------------------------------------------
// r^-n for the stage from 1/r^2 and 1/r^6
__device__ __forceinline__ double inv_rn64(const StageDev &st, double r2, double ir2, double ir6)
{
    if (st.nkind == 1) {
        // factor by factor: r^-12 as the square of r^-6 would double that one's rounding
        const int n = st.nint, h = n >> 1;
        double p = n >= 6 ? ir6 : 1.0;
        for (int k = n >= 6 ? 3 : 0; k < h; ++k) p *= ir2;
        if (n & 1) p *= rsqrt(r2);
        return p;
    }
    if (st.nkind == 2) return ir6 * sqrt(sqrt(sqrt(r2)));
    if (st.nkind == 3) return ir6 * sqrt(rsqrt(r2));
    return exp2(-0.5 * st.n * log2(r2));
}

__device__ __forceinline__ double mlj_fr64(const StageDev &st, double r2, double ir2)
{
    const double ir6 = ir2 * ir2 * ir2;
    return (6.0 * st.c2 * ir6 - st.n * st.c1 * inv_rn64(st, r2, ir2, ir6)) * ir2;
}

__device__ __forceinline__ void add64(double a, double3 x, double3 &F)
{
    F.x += a * x.x;
    F.y += a * x.y;
    F.z += a * x.z;
}

// One Newton step each, two to four operations of the pipe, where a divide or
// another square root is a dozen: 1 / l from q = 1 / l to a few ulps, 1 / sqrt(l)
// likewise, a / b from r = 1 / b rounded.  The results are within an ulp, as those
// of the instructions' sequences that they stand for.
__device__ __forceinline__ double better_inv(double l, double q) { return fma(q, fma(-l, q, 1.0), q); }
__device__ __forceinline__ double better_rsqrt(double l, double i) { return fma(0.5 * i, fma(-l * i, i, 1.0), i); }
__device__ __forceinline__ double better_div(double a, double b, double r)
{
    const double t = a * r;
    return fma(fma(-t, b, a), r, t);
}

// Bond (Eq. 10) and bending (Eq. 4) forces from the chain partners bp = (s-2, s-1, s+1, s+2)
__device__ __forceinline__ void bonded64(const GeoF64 &g, const StageDev &st, double kap, double rc2, int4 bp,
                                         double3 &F, unsigned &err)
{
    const bool hm2 = bp.x >= 0, hm1 = bp.y >= 0, hp1 = bp.z >= 0, hp2 = bp.w >= 0;
    double3 Bm2 = make_double3(0., 0., 0.), Bm1 = Bm2, B0 = Bm2, Bp1 = Bm2;     // bonds s-2, s-1, s, s+1
    double3 rm1 = Bm2;
    if (hm1) {
        rm1 = g.rel(bp.y);
        Bm1 = make_double3(-rm1.x, -rm1.y, -rm1.z);
        if (hm2 && kap != 0.0) Bm2 = sub3(rm1, g.rel(bp.x));
    }
    if (hp1) {
        B0 = g.rel(bp.z);
        if (hp2 && kap != 0.0) Bp1 = sub3(g.rel(bp.w), B0);
    }
    const double l1 = dot3(Bm1, Bm1), l2 = dot3(B0, B0);
    const double i1 = rsqrt(l1), i2 = rsqrt(l2);                                // infinite past a chain end, unused
    const double q1 = better_inv(l1, i1 * i1), q2 = better_inv(l2, i2 * i2);
    const double invR0sq = 1.0 / st.R0sq;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        if (side == 0 ? hm1 : hp1) {
            const double r2 = side == 0 ? l1 : l2;
            double q = 1.0 - better_div(r2, st.R0sq, invR0sq), fr;
            if (st.qmin > 0.0 && q < st.qmin) {          // continuation beyond r* (kg_params.fene_qmin)
                fr = st.kfene / st.qmin;
                if (!(r2 < 4.0 * st.R0sq)) err |= ERR_OVERSTRETCH;
            } else {
                if (!(r2 < st.R0sq)) err |= ERR_OVERSTRETCH;
                q = fmax(q, 1e-6);                       // finite even when flagged
                fr = st.kfene / q;
            }
            if (r2 < rc2) fr += mlj_fr64(st, r2, side == 0 ? q1 : q2);
            add64(fr, side == 0 ? rm1 : B0, F);
        }
    }
    if (kap != 0.0) {
        if (hm1 && hp1) {                    // vertex s: force kappa (g1 - g2)
            const double inv = better_rsqrt(l1 * l2, i1 * i2), cs = dot3(Bm1, B0) * inv;
            add64(kap * (inv + cs * q2), B0, F);
            add64(-kap * (inv + cs * q1), Bm1, F);
        }
        if (hp2) {                           // vertex s+1, s is its first end: -kappa g1
            const double l3 = dot3(Bp1, Bp1), inv = better_rsqrt(l2 * l3, i2 * rsqrt(l3)), cs = dot3(B0, Bp1) * inv;
            add64(-kap * inv, Bp1, F);
            add64(kap * cs * q2, B0, F);
        }
        if (hm2) {                           // vertex s-1, s is its last end: +kappa g2
            const double l0 = dot3(Bm2, Bm2), inv = better_rsqrt(l0 * l1, i1 * rsqrt(l0)), cs = dot3(Bm2, Bm1) * inv;
            add64(kap * inv, Bm2, F);
            add64(-kap * cs * q1, Bm1, F);
        }
    }
}

constexpr int F64_BLOCK = 64;
constexpr int F64_PAIRS = 192;           // near pairs of a warp that one round takes (mean about 110)

__global__ void __launch_bounds__(F64_BLOCK) k_step_f64(const SimDev *__restrict__ Sp, const StageDev *__restrict__ stp,
                                                 double *__restrict__ x, double *__restrict__ u,
                                                 const double4_32a *__restrict__ pcur, double4_32a *__restrict__ pnext,
                                                 const double4_32a *__restrict__ xb, const float4 *__restrict__ recb,
                                                 const float4 *__restrict__ gcur, float4 *__restrict__ gnext,
                                                 const unsigned *__restrict__ nl,
                                                 const int *__restrict__ nn, const int *__restrict__ slot_of,
                                                 const int4 *__restrict__ bp, unsigned *__restrict__ flags,
                                                 const long long *__restrict__ stepp, LoopDev *loop, int kstep)
{
    __shared__ unsigned stop;
    if (threadIdx.x == 0) stop = step_off(flags, loop, kstep);
    __syncthreads();
    if (stop) return;
    const SimDev &S = *Sp;
    const StageDev &st = *stp;
    const long long step = *stepp + (loop ? 1 + kstep : 0);
    __shared__ double pf_s[F64_BLOCK / 32][4 * F64_PAIRS];       // (dU/dr)/r and the vector of each pair
    __shared__ unsigned pair_s[F64_BLOCK / 32][F64_PAIRS];
    const int s = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    double *const pf = pf_s[threadIdx.x >> 5];
    unsigned *const pair = pair_s[threadIdx.x >> 5];
    bool rebuild = false;
    unsigned err = 0;
    const bool live = s < S.M;
    const int cnt = live ? __ldg(nn + s) : 0;
    const int kmax = __reduce_max_sync(0xffffffffu, cnt);
    double3 F = make_double3(0., 0., 0.);
    {
        const int slot = __ldg(slot_of + (live ? s : 0));
        const MeltDev &md = S.melt[melt_of(S, slot)];
        const unsigned *__restrict__ col = nl + s;
        const float4 gi = __ldg(gcur + (live ? s : 0));
        const float h = md.hf, near2 = md.near2;
        for (int k0 = 0; k0 < kmax; k0 += 32) {
            unsigned mask = 0;
            const int kn = min(32, cnt - k0);
            for (int k = 0; k < kn; k += 4) {
                unsigned e[4];
                float4 p[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) e[i] = __ldg(col + (size_t)(k0 + min(k + i, kn - 1)) * S.Mp);
#pragma unroll
                for (int i = 0; i < 4; ++i) p[i] = __ldg(gcur + (e[i] & IDX_MASK));
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int q = (int)(e[i] >> IDX_BITS);
                    const float dx = fmaf((float)(q % 3 - 1), h, p[i].x - gi.x);
                    const float dy = fmaf((float)((q / 3) % 3 - 1), h, p[i].y - gi.y);
                    const float dz = fmaf((float)(q / 9 - 1), h, p[i].z - gi.z);
                    const bool close = fmaf(dz, dz, fmaf(dy, dy, dx * dx)) < near2;
                    mask |= (unsigned)(close && k + i < kn) << (k + i);
                }
            }
            // the warp's near pairs in order of lane and list: this lane's are [first, first + n)
            const int n = __popc(mask);
            int first = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, first, o);
                if (lane >= o) first += t;
            }
            const int total = __shfl_sync(0xffffffffu, first, 31);
            first -= n;
            for (int b = 0; b < total; b += F64_PAIRS) {
                unsigned left = mask;
                for (int i = first - b; left; ++i) {
                    const int k = __ffs(left) - 1;
                    left &= left - 1;
                    if (i >= 0 && i < F64_PAIRS)
                        pair[i] = (__ldg(col + (size_t)(k0 + k) * S.Mp) & IDX_MASK) | ((unsigned)lane << IDX_BITS);
                }
                __syncwarp();
                for (int i = lane; i < min(F64_PAIRS, total - b); i += 32) {
                    const int own = s - lane + (int)(pair[i] >> IDX_BITS);
                    const MeltDev &mo = S.melt[melt_of(S, __ldg(slot_of + own))];
                    GeoF64 g{pcur, mo.L, mo.invL, {}};
                    g.self(own);
                    const double3 d = g.rel((int)(pair[i] & IDX_MASK));
                    const double r2 = dot3(d, d);
                    const double fr = r2 < S.rc2 ? mlj_fr64(st, r2, 1.0 / r2) : 0.0;
                    pf[i] = fr;
                    pf[F64_PAIRS + i] = d.x;
                    pf[2 * F64_PAIRS + i] = d.y;
                    pf[3 * F64_PAIRS + i] = d.z;
                }
                __syncwarp();
                for (int i = max(first - b, 0); i < min(first + n - b, F64_PAIRS); ++i) {
                    const double fr = pf[i];
                    add64(fr, make_double3(pf[F64_PAIRS + i], pf[2 * F64_PAIRS + i], pf[3 * F64_PAIRS + i]), F);
                }
                __syncwarp();
            }
        }
    }
    if (live) {
        const int slot = __ldg(slot_of + s);
        const int m = melt_of(S, slot);
        const MeltDev &md = S.melt[m];
        const int rel = slot - md.off;
        GeoF64 g{pcur, md.L, md.invL, {}};
        g.self(s);
        const int Mp = S.Mp;
        bonded64(g, st, md.kappa, S.rc2, __ldg(bp + s), F, err);
        const double3 gn = gauss3_d(draw(S.seed, m, 0, (unsigned long long)step, (uint32_t)rel));
        double3 v = make_double3(u[s], u[Mp + s], u[2 * Mp + s]);
        v.x += st.dt * (F.x - st.gamma * v.x + st.amp * gn.x);
        v.y += st.dt * (F.y - st.gamma * v.y + st.amp * gn.y);
        v.z += st.dt * (F.z - st.gamma * v.z + st.amp * gn.z);
        u[s] = v.x; u[Mp + s] = v.y; u[2 * Mp + s] = v.z;
        const double nx = x[s] + st.dt * v.x, ny = x[Mp + s] + st.dt * v.y, nz = x[2 * Mp + s] + st.dt * v.z;
        x[s] = nx; x[Mp + s] = ny; x[2 * Mp + s] = nz;
        pnext[s] = make_double4_32a(nx, ny, nz, 0.0);
        const double4_32a b = xb[s];
        const float dx = (float)(nx - b.x), dy = (float)(ny - b.y), dz = (float)(nz - b.z);
        const float4 rb = __ldg(recb + s);
        gnext[s] = make_float4(rb.x + dx, rb.y + dy, rb.z + dz, rb.w);
        // a little early: the binary32 displacement is good to a few 2^-24
        rebuild = !(fmaf(dz, dz, fmaf(dy, dy, dx * dx)) <= S.half_skin2f * (1.0f - 1e-6f));
        if (!isfinite(v.x + v.y + v.z)) err |= ERR_NONFINITE;
    }
    if (__syncthreads_or(rebuild) && threadIdx.x == 0) {
        if (loop) atomicOr(&loop->req, 1u << kstep);
        else atomicOr(flags + 1, 1u);
    }
    if (err) atomicOr(flags, err);
}

// ---------------------------------------------------------------------------
// rebuild chain: each kernel returns at once unless flags[1] requests a
// rebuild; the last block of k_nlist to finish clears the request
// ---------------------------------------------------------------------------
// build records (offset from the Verlet-cell corner + cell coordinates),
// gather buffers reset, Verlet-grid cell + rank within it
__global__ void __launch_bounds__(256) k_bin_md(const SimDev *__restrict__ Sp, double *__restrict__ x,
                                               double *__restrict__ xb64,
                                               float4 *__restrict__ recb, float4 *dcur,
                                               float4 *__restrict__ pgcur, double4_32a *__restrict__ pcur,
                                               double4_32a *__restrict__ xb, int *__restrict__ cellid,
                                               int *__restrict__ rank, int *__restrict__ count,
                                               const int *__restrict__ slot_of, unsigned *__restrict__ flags,
                                               const float4 *dother, const LoopDev *__restrict__ loop)
{
    if (!flags[1] || flags[0]) return;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= Sp->M) return;
    const unsigned err =
        bin_md_one(*Sp, s, x, xb64, recb, loop && loop->src ? dother : dcur, dcur, pgcur, pcur, xb, cellid, rank, count,
                   slot_of);                       // a loop's pass starts in buffer 0 wherever the last one ended
    if (err) atomicOr(flags, err);
}

// DB grid: cell of each particle from its wrapped position (cells >= 1.3
// sigma), and its binary32 record (offset from the cell corner, cell
// coordinates) for the swap-bond prefilter
__global__ void __launch_bounds__(256) k_bin_db(const SimDev *__restrict__ Sp, const double *__restrict__ x,
                                               int *__restrict__ cellid, int *__restrict__ rank,
                                               int *__restrict__ count, const int *__restrict__ slot_of,
                                               float4 *__restrict__ rec)
{
    const SimDev &S = *Sp;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= S.M) return;
    const MeltDev &md = S.melt[melt_of(S, slot_of[s])];
    int cell[3];
    float off[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) cell[d] = cell_of(x[d * S.Mp + s], md.hdb, md.invhdb, md.ndb, off[d]);
    rec[s] = make_float4(off[0], off[1], off[2], __uint_as_float(pack_code(cell[0], cell[1], cell[2])));
    const int c = md.dbcell_off + (cell[2] * md.ndb + cell[1]) * md.ndb + cell[0];
    cellid[s] = c;
    rank[s] = atomicAdd(count + c, 1);
}

// exclusive scan, phase 1: per 1024-element block, local scan + block total
__global__ void __launch_bounds__(1024) k_scan1(const int *__restrict__ in, int *__restrict__ out,
                                               int *__restrict__ bsum, int n, const unsigned *__restrict__ flags)
{
    if (flags && (!flags[1] || flags[0])) return;
    __shared__ int wsum[32];
    const int i = blockIdx.x * 1024 + threadIdx.x;
    const int v = i < n ? in[i] : 0;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    if (w == 0) {
        int ws = wsum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, ws, o);
            if (lane >= o) ws += t;
        }
        wsum[lane] = ws;
    }
    __syncthreads();
    const int base = w ? wsum[w - 1] : 0;
    if (i < n) out[i] = base + incl - v;
    if (threadIdx.x == 1023) bsum[blockIdx.x] = base + incl;
}

// phase 2: add the totals of all preceding blocks; out[n] = grand total
__global__ void __launch_bounds__(1024) k_scan2(int *__restrict__ out, const int *__restrict__ bsum, int n,
                                               int nblk, const unsigned *__restrict__ flags)
{
    if (flags && (!flags[1] || flags[0])) return;
    __shared__ int off_s;
    if (threadIdx.x < 32) {
        int acc = 0;
        for (int b = threadIdx.x; b < (int)blockIdx.x; b += 32) acc += bsum[b];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if (threadIdx.x == 0) off_s = acc;
    }
    __syncthreads();
    const int i = blockIdx.x * 1024 + threadIdx.x;
    if (i < n) out[i] += off_s;
    if (blockIdx.x == nblk - 1 && threadIdx.x == 0) {
        int tot = 0;
        for (int b = 0; b < nblk; ++b) tot += bsum[b];
        out[n] = tot;
    }
}

// slot list in cell order; with recb, the build offsets are copied into the
// same order (recs, w = the compute index) so that a cell's candidates are one
// contiguous run of single 16-byte loads
__global__ void __launch_bounds__(256) k_scatter(const int *__restrict__ cellid, const int *__restrict__ rank,
                                                const int *__restrict__ start, int *__restrict__ list, int M,
                                                const unsigned *__restrict__ flags)
{
    if (flags && (!flags[1] || flags[0])) return;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < M) scatter_one(s, cellid, rank, start, list);
}

// within-cell order by compute index (deterministic lists), the records in
// the same order, the counts cleared (cellrank_one, kg_rebuild.cuh)
__global__ void __launch_bounds__(256) k_cellrank(const int *__restrict__ cellid, const int *__restrict__ start,
                                                 const int *__restrict__ tmp, int *__restrict__ list,
                                                 const float4 *__restrict__ recb, float4 *__restrict__ recs,
                                                 int *__restrict__ count, int M, unsigned *__restrict__ flags)
{
    if (!flags[1] || flags[0]) return;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < M && cellrank_one(p, cellid, start, tmp, list, recb, recs, count)) atomicOr(flags, ERR_NL_CAPACITY);
}

// Verlet-list build (the per-monomer work is nlist_one, kg_rebuild.cuh).
// The last block to finish clears the rebuild request.
// (256, 5): at most 48 registers and no spills; more resident warps hide the
// candidate loads (tighter caps spill, looser ones leave the SM half idle)
constexpr int NL_BLOCK = 256;

__global__ void __launch_bounds__(NL_BLOCK, 5) k_nlist(const __grid_constant__ NlArgs A)
{
    __shared__ unsigned go;
    if (threadIdx.x == 0) go = (A.flags[1] && !A.flags[0]) ? 1u : 0u;
    __syncthreads();
    if (!go) return;                                         // block-uniform
    const int s = blockIdx.x * NL_BLOCK + threadIdx.x;
    const unsigned err = nlist_one<true>(A, s);
    if (err) atomicOr(A.flags, err);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(A.flags + 4, 1u) == gridDim.x - 1) {
            A.flags[1] = 0u;
            A.flags[4] = 0u;
            A.flags[5] += 1u;                    // Verlet builds completed
            A.flags[RES_BUILT] = 0u;             // the cell order is in clist
        }
    }
}

// ---------------------------------------------------------------------------
// forces + energies (observables, parity): F_c written as binary64; per block
// partial sums [pair, bond, angle, virial, kinetic] in binary64, where the
// kinetic part uses v_n = u + dt/2 (F_c - gamma u + amp g_n).
// ---------------------------------------------------------------------------
template <class G>
__global__ void __launch_bounds__(128) k_forces(const SimDev *__restrict__ Sp, const StageDev *__restrict__ stp,
                                               G g, const void *__restrict__ uptr, int lo, int hi,
                                               const unsigned *__restrict__ nl, const int *__restrict__ nn,
                                               const int *__restrict__ slot_of, const int4 *__restrict__ bp,
                                               double *__restrict__ Fout, double *__restrict__ part,
                                               unsigned *__restrict__ flags, long long step)
{
    using T = typename G::T;
    const SimDev &S = *Sp;
    const StageDev &st = *stp;
    const int s = lo + blockIdx.x * blockDim.x + threadIdx.x;
    double e[5] = {0, 0, 0, 0, 0};
    unsigned err = 0;
    if (s < hi) {
        const int slot = slot_of[s];
        const int m = melt_of(S, slot);
        const MeltDev &md = S.melt[m];
        const int rel = slot - md.off;
        G gg = g;
        gg.melt(md, m);
        gg.self(s);
        const auto F = force_on(gg, S, st, md, s, bp[s], nl, __ldg(nn + s), e, err);
        const int Mp = S.Mp;
        if (Fout) {
            Fout[s] = (double)F.x; Fout[Mp + s] = (double)F.y; Fout[2 * Mp + s] = (double)F.z;
        }
        const double3 gn = gauss3_d(draw(S.seed, m, 0, (unsigned long long)step, (uint32_t)rel));
        const T *u = (const T *)uptr;
        const double ux = (double)u[s], uy = (double)u[Mp + s], uz = (double)u[2 * Mp + s];
        const double vx = ux + 0.5 * st.dt * ((double)F.x - st.gamma * ux + st.amp * gn.x);
        const double vy = uy + 0.5 * st.dt * ((double)F.y - st.gamma * uy + st.amp * gn.y);
        const double vz = uz + 0.5 * st.dt * ((double)F.z - st.gamma * uz + st.amp * gn.z);
        e[4] = 0.5 * (vx * vx + vy * vy + vz * vz);
    }
    if (err) atomicOr(flags, err);
    // deterministic block reduction (fixed tree)
    __shared__ double sh[5][128];
#pragma unroll
    for (int k = 0; k < 5; ++k) sh[k][threadIdx.x] = e[k];
    __syncthreads();
    for (int w = 64; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
#pragma unroll
            for (int k = 0; k < 5; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < 5; ++k) part[blockIdx.x * 5 + k] = sh[k][0];
}

// ---------------------------------------------------------------------------
// compute order: chain partners, re-sorting, and gathers back to slot order
// ---------------------------------------------------------------------------
// bp[i] = compute indices of slots s-2, s-1, s+1, s+2 of i's chain (-1 past an end)
__global__ void __launch_bounds__(256) k_bonded(const SimDev *__restrict__ Sp, const int *__restrict__ slot_of,
                                               const int *__restrict__ comp_of, int4 *__restrict__ bp)
{
    const SimDev &S = *Sp;
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= S.M) return;
    const int s = slot_of[j];
    const MeltDev &md = S.melt[melt_of(S, s)];
    const int i = (s - md.off) % md.N, N = md.N;
    bp[j] = make_int4(i >= 2 ? comp_of[s - 2] : -1, i >= 1 ? comp_of[s - 1] : -1,
                      i <= N - 2 ? comp_of[s + 1] : -1, i <= N - 3 ? comp_of[s + 2] : -1);
}

// New compute order = the cell order of the last Verlet build (clist): gather
// the per-monomer state into scratch ...
template <typename U>
__global__ void __launch_bounds__(256) k_sort_gather(int M, int Mp, const int *__restrict__ order,
                                                    const double *__restrict__ x, const U *__restrict__ u,
                                                    const int *__restrict__ pid, const int *__restrict__ slot_of,
                                                    double *__restrict__ sx, U *__restrict__ su,
                                                    int *__restrict__ spid, int *__restrict__ sslot)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= M) return;
    const int o = order[j];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        sx[d * Mp + j] = x[d * Mp + o];
        su[d * Mp + j] = u[d * Mp + o];
    }
    spid[j] = pid[o];
    sslot[j] = slot_of[o];
}

// ... and copy it back, with the inverse map.
template <typename U>
__global__ void __launch_bounds__(256) k_sort_finish(int M, int Mp, double *__restrict__ x, U *__restrict__ u,
                                                    int *__restrict__ pid, int *__restrict__ slot_of,
                                                    int *__restrict__ comp_of, const double *__restrict__ sx,
                                                    const U *__restrict__ su, const int *__restrict__ spid,
                                                    const int *__restrict__ sslot)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= M) return;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        x[d * Mp + j] = sx[d * Mp + j];
        u[d * Mp + j] = su[d * Mp + j];
    }
    pid[j] = spid[j];
    const int s = sslot[j];
    slot_of[j] = s;
    comp_of[s] = j;
}

// out[d][r] = in[d][comp_of[off + r]] for r < n: slot order for the caller
__global__ void __launch_bounds__(256) k_to_slots(const double *__restrict__ in, int in_stride,
                                                 const int *__restrict__ comp_of, int off, int n,
                                                 double *__restrict__ out, int out_stride, int dims)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int j = comp_of[off + r];
    for (int d = 0; d < dims; ++d) out[(size_t)d * out_stride + r] = in[(size_t)d * in_stride + j];
}

// State of a melt in slot order, in one pass: positions, velocities (binary32
// state widened) and ids, each where asked for (null: not).
template <typename U>
__global__ void __launch_bounds__(256) k_state_to_slots(const double *__restrict__ x, const U *__restrict__ u,
                                                       const int *__restrict__ pid, int Mp,
                                                       const int *__restrict__ comp_of, int off, int n,
                                                       double *__restrict__ xo, double *__restrict__ uo,
                                                       int *__restrict__ po)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int j = comp_of[off + r];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        if (xo) xo[(size_t)d * n + r] = x[(size_t)d * Mp + j];
        if (uo) uo[(size_t)d * n + r] = (double)u[(size_t)d * Mp + j];
    }
    if (po) po[r] = pid[j];
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static inline int nblk(long long n, int b) { return (int)((n + b - 1) / b); }

void bonded_partners(kg_ctx *c)
{
    ++c->launches;
    k_bonded<<<nblk(c->M, 256), 256, 0, c->stream>>>(c->d_sim, c->slot_of, c->comp_of, c->bp);
}

// Re-sort the per-monomer state into the cell order of the last Verlet build.
// The list then refers to the old order, so a rebuild is requested.
void md_sort(kg_ctx *c)
{
    md_materialize(c);
    resident_cell_order(c);
    const int Mp = c->Mp;
    double *sx = c->scratch;
    int *spid = (int *)(c->scratch + 6 * (size_t)Mp);
    int *sslot = spid + Mp;
    c->launches += 2;
    if (c->precision == KG_MIXED) {
        float *su = (float *)(c->scratch + 3 * (size_t)Mp);
        k_sort_gather<float><<<nblk(c->M, 256), 256, 0, c->stream>>>(c->M, Mp, c->clist, c->x, (const float *)c->u,
                                                                    c->pid, c->slot_of, sx, su, spid, sslot);
        k_sort_finish<float><<<nblk(c->M, 256), 256, 0, c->stream>>>(c->M, Mp, c->x, (float *)c->u, c->pid,
                                                                    c->slot_of, c->comp_of, sx, su, spid, sslot);
    } else {
        double *su = c->scratch + 3 * (size_t)Mp;
        k_sort_gather<double><<<nblk(c->M, 256), 256, 0, c->stream>>>(c->M, Mp, c->clist, c->x,
                                                                     (const double *)c->u, c->pid, c->slot_of, sx,
                                                                     su, spid, sslot);
        k_sort_finish<double><<<nblk(c->M, 256), 256, 0, c->stream>>>(c->M, Mp, c->x, (double *)c->u, c->pid,
                                                                     c->slot_of, c->comp_of, sx, su, spid, sslot);
    }
    if (c->precision == KG_MIXED) {    // sorted current positions become the build positions
        cudaMemcpyAsync(c->xb64, c->x, 3 * (size_t)Mp * sizeof(double), cudaMemcpyDeviceToDevice, c->stream);
        cudaMemsetAsync(c->dlt[c->cur], 0, (size_t)Mp * sizeof(float4), c->stream);
    }
    msd_permute(c, c->clist);
    bonded_partners(c);
    static const unsigned one = 1u;
    cudaMemcpyAsync(c->flags + 1, &one, sizeof(unsigned), cudaMemcpyHostToDevice, c->stream);
}

// mixed: current binary64 positions x = xb64 + dlt[cur] (the same sum as the
// build's fold, so a later build finds the same values)
__global__ void __launch_bounds__(256) k_materialize(double *__restrict__ x, const double *__restrict__ xb64,
                                                    const float4 *__restrict__ d, int M, int Mp)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= M) return;
    const float4 e = d[s];
    x[s] = xb64[s] + (double)e.x;
    x[Mp + s] = xb64[Mp + s] + (double)e.y;
    x[2 * Mp + s] = xb64[2 * Mp + s] + (double)e.z;
}

void md_materialize(kg_ctx *c)
{
    if (c->precision != KG_MIXED) return;
    ++c->launches;
    k_materialize<<<nblk(c->M, 256), 256, 0, c->stream>>>(c->x, c->xb64, c->dlt[c->cur], c->M, c->Mp);
}

void to_slots(kg_ctx *c, int melt, const double *in_comp, double *out_dev, int dims)
{
    const MeltDev &md = c->sim.melt[melt];
    ++c->launches;
    k_to_slots<<<nblk(md.M, 256), 256, 0, c->stream>>>(in_comp, c->Mp, c->comp_of, md.off, md.M, out_dev, md.M,
                                                       dims);
}

void state_to_slots(kg_ctx *c, int melt, double *x_dev, double *u_dev, int *pid_dev)
{
    const MeltDev &md = c->sim.melt[melt];
    ++c->launches;
    const int nb = nblk(md.M, 256);
    if (c->precision == KG_MIXED)
        k_state_to_slots<float><<<nb, 256, 0, c->stream>>>(c->x, (const float *)c->u, c->pid, c->Mp, c->comp_of, md.off,
                                                           md.M, x_dev, u_dev, pid_dev);
    else
        k_state_to_slots<double><<<nb, 256, 0, c->stream>>>(c->x, (const double *)c->u, c->pid, c->Mp, c->comp_of,
                                                            md.off, md.M, x_dev, u_dev, pid_dev);
}

// First kernel of a directly launched MD step: advance the device step counter
// (the index of the step about to run).
__global__ void k_begin_step(long long *__restrict__ stepp) { stepp[0] += 1; }

__global__ void k_set_step(long long *__restrict__ stepp, long long v) { stepp[0] = v; }

void scan_counts(kg_ctx *c, const int *count, int *start, int n, int *bsum)
{
    const int nb = nblk(n, 1024);
    k_scan1<<<nb, 1024, 0, c->stream>>>(count, start, bsum, n, nullptr);
    k_scan2<<<nb, 1024, 0, c->stream>>>(start, bsum, n, nb, nullptr);
}

static void launch_rebuild(kg_ctx *c, cudaStream_t st, int cur, LoopDev *loop);

void rebuild_md(kg_ctx *c)
{
    c->launches += 6;
    launch_rebuild(c, c->stream, c->cur, nullptr);
}

NlArgs nl_args(const kg_ctx *c)
{
    NlArgs a{};
    a.x = c->x;
    a.recb = c->recb;
    a.recs = c->recs;
    a.start = c->cstart;
    a.nl = c->nl;
    a.nn = c->nn;
    a.flags = c->flags;
    a.slot_of = c->slot_of;
    a.bp = c->bp;
    a.M = c->M;
    a.Mp = c->Mp;
    a.maxnb = c->maxnb;
    a.n_melts = c->sim.n_melts;
    a.rl2 = c->sim.rl2;
    for (int m = 0; m < c->sim.n_melts; ++m) {
        const MeltDev &md = c->sim.melt[m];
        a.melt[m] = MeltNl{md.off, md.cell_off, md.nbk, md.nc, md.hf, md.nl_lo, md.nl_hi, md.invLf, md.L};
    }
    return a;
}

static void launch_rebuild(kg_ctx *c, cudaStream_t st, int cur, LoopDev *loop)
{
    const bool mixed = c->precision == KG_MIXED;
    k_bin_md<<<nblk(c->M, 256), 256, 0, st>>>(c->d_sim, c->x, mixed ? c->xb64 : nullptr, c->recb,
                                              mixed ? c->dlt[cur] : nullptr, c->pg[cur], mixed ? nullptr : c->pos64[cur],
                                              c->xb, c->cellid, c->rank, c->ccount, c->slot_of, c->flags,
                                              mixed ? c->dlt[cur ^ 1] : nullptr, loop);
    const int nb = nblk(c->ncell_md, 1024);
    k_scan1<<<nb, 1024, 0, st>>>(c->ccount, c->cstart, c->bsum, c->ncell_md, c->flags);
    k_scan2<<<nb, 1024, 0, st>>>(c->cstart, c->bsum, c->ncell_md, nb, c->flags);
    k_scatter<<<nblk(c->M, 256), 256, 0, st>>>(c->cellid, c->rank, c->cstart, c->ctmp, c->M, c->flags);
    k_cellrank<<<nblk(c->M, 256), 256, 0, st>>>(c->cellid, c->cstart, c->ctmp, c->clist, c->recb, c->recs, c->ccount,
                                                c->M, c->flags);
    k_nlist<<<nblk(c->M, NL_BLOCK), NL_BLOCK, 0, st>>>(nl_args(c));
}

static void launch_step_kernel(kg_ctx *c, cudaStream_t st, int cur, LoopDev *loop, int k)
{
    if (c->precision == KG_MIXED) {
        step_mixed_launch(c, st, cur, loop, k);
        return;
    }
    k_step_f64<<<nblk(c->M, F64_BLOCK), F64_BLOCK, 0, st>>>(c->d_sim, c->d_stage, c->x, (double *)c->u, c->pos64[cur], c->pos64[cur ^ 1],
                                        c->xb, c->recb, c->pg[cur], c->pg[cur ^ 1], c->nl, c->nn, c->slot_of, c->bp, c->flags, c->d_step, loop, k);
}

// Captured graphs hold the step kernel's by-value arguments (stage
// parameters among them): drop them when those change.
void graphs_reset(kg_ctx *c)
{
    for (cudaGraphExec_t &e : c->gexec) {
        if (e) cudaGraphExecDestroy(e);
        e = nullptr;
    }
}

void set_device_step(kg_ctx *c, long long v)
{
    ++c->launches;
    k_set_step<<<1, 1, 0, c->stream>>>(c->d_step, v);
}

// One MD step: the Verlet list is rebuilt first if the previous step (or a
// configuration load or an accepted swap) asked for it.
void prof_collect(kg_ctx *c)
{
    if (!c->ev_used) return;
    cudaStreamSynchronize(c->stream);
    for (int i = 0; i < c->ev_used; ++i) {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, c->ev[2 * i], c->ev[2 * i + 1]);
        c->prof_ms += ms;
    }
    c->prof_n += c->ev_used;
    c->ev_used = 0;
}

void md_step(kg_ctx *c)
{
    k_begin_step<<<1, 1, 0, c->stream>>>(c->d_step);
    ++c->launches;
    rebuild_md(c);
    cudaEvent_t e1 = nullptr;
    if (c->prof_on) {
        if (c->ev.empty()) {
            c->ev.resize(2 * 1024);
            for (auto &e : c->ev) cudaEventCreate(&e);
        }
        if (2 * c->ev_used >= (int)c->ev.size()) prof_collect(c);
        cudaEventRecord(c->ev[2 * c->ev_used], c->stream);
        e1 = c->ev[2 * c->ev_used + 1];
        ++c->ev_used;
    }
    ++c->launches;
    launch_step_kernel(c, c->stream, c->cur, nullptr, 0);
    if (e1) cudaEventRecord(e1, c->stream);
    c->cur ^= 1;
}

// ---------------------------------------------------------------------------
// captured step loop: a graph with one while node, whose body is the rebuild
// chain (its kernels return at once without a request), up to LOOP_MAX step
// kernels and a one-thread kernel that ends the pass.  A step that asks for a
// rebuild sets its bit; the later steps of the pass see it and return at once,
// and the next pass starts with the chain.  So the graph's control (a while
// node's turn, ~10 us) is paid once per list build, where a conditional node
// in front of every step cost about 13 us a step (the step kernel of 200,000
// monomers takes 14, that of 1.6M 91).  The body is as long as the measured
// number of steps between builds, so few step kernels are launched in vain.
// Passes start in buffer 0 (a build writes it, and the body's length is even);
// k_loop_settle moves the result there when the last pass ended in buffer 1.
// ---------------------------------------------------------------------------
__global__ void k_loop_begin(LoopDev *lp, long long steps, int len)
{
    lp->rem = steps;
    lp->n = (int)(steps < len ? steps : len);
    lp->src = lp->par = 0;
    lp->req = 0u;
}

__global__ void k_loop_end(LoopDev *lp, int len, long long *__restrict__ stepp, unsigned *__restrict__ flags,
                           cudaGraphConditionalHandle h)
{
    const bool more = loop_finish(lp, len, stepp, flags);
    cudaGraphSetConditional(h, more ? 1u : 0u);
}

void loop_begin(cudaStream_t st, LoopDev *lp, long long steps, int len) { k_loop_begin<<<1, 1, 0, st>>>(lp, steps, len); }

__global__ void __launch_bounds__(256) k_loop_settle(const LoopDev *__restrict__ lp, bool always,
                                                    float4 *__restrict__ a0, const float4 *__restrict__ a1, int na,
                                                    float4 *__restrict__ b0, const float4 *__restrict__ b1, int nb)
{
    if (!always && !lp->par) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < na; i += gridDim.x * blockDim.x) a0[i] = a1[i];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nb; i += gridDim.x * blockDim.x) b0[i] = b1[i];
}

bool capture_loop(cudaStream_t s, cudaGraphExec_t *exec, const std::function<void(cudaGraphConditionalHandle)> &pass)
{
    cudaGraph_t g = nullptr;
    *exec = nullptr;
    if (cudaGraphCreate(&g, 0) != cudaSuccess) return false;
    cudaGraphConditionalHandle h;
    bool ok = cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault) == cudaSuccess;
    cudaGraphNodeParams cp{};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = h;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t cn;
    ok = ok && cudaGraphAddNode(&cn, g, nullptr, nullptr, 0, &cp) == cudaSuccess;
    if (ok) {
        cudaGraph_t body = cp.conditional.phGraph_out[0];
        ok = cudaStreamBeginCaptureToGraph(s, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal) ==
             cudaSuccess;
        if (ok) {
            pass(h);
            ok = cudaStreamEndCapture(s, &body) == cudaSuccess && cudaGetLastError() == cudaSuccess;
        }
    }
    ok = ok && cudaGraphInstantiate(exec, g, 0) == cudaSuccess;
    cudaGraphDestroy(g);
    if (!ok) {
        cudaGetLastError();
        *exec = nullptr;
    }
    return ok;
}

// buffer 1 of the state that alternates between steps to buffer 0
static void loop_settle(kg_ctx *c, bool always)
{
    const bool mixed = c->precision == KG_MIXED;
    ++c->launches;
    k_loop_settle<<<std::min(nblk(c->M, 256), 152 * 8), 256, 0, c->stream>>>(
        c->loop, always, mixed ? c->dlt[0] : (float4 *)c->pos64[0], mixed ? c->dlt[1] : (const float4 *)c->pos64[1],
        mixed ? c->M : 2 * c->M, c->pg[0], c->pg[1], c->M);
}

bool md_loop_steps(kg_ctx *c, int n)
{
    if (c->graph_failed) return false;
    // the multiple of four at or above the measured number of steps between builds
    int q = 0;
    while (4 * (q + 1) < LOOP_MAX && c->build_every > 4.0 * (q + 1)) ++q;
    const int len = 4 * (q + 1);
    if (!c->gexec[q]) {
        if (!c->cap_stream && cudaStreamCreateWithFlags(&c->cap_stream, cudaStreamNonBlocking) != cudaSuccess) {
            c->graph_failed = true;
            return false;
        }
        const cudaStream_t s = c->cap_stream;
        if (!capture_loop(s, &c->gexec[q], [&](cudaGraphConditionalHandle h) {
                launch_rebuild(c, s, 0, c->loop);
                for (int k = 0; k < len; ++k) launch_step_kernel(c, s, k & 1, c->loop, k);
                k_loop_end<<<1, 1, 0, s>>>(c->loop, len, c->d_step, c->flags, h);
            })) {
            c->graph_failed = true;
            return false;
        }
    }
    loop_begin(c->stream, c->loop, n, len);
    if (c->cur) loop_settle(c, true);          // after an odd number of direct steps: start from buffer 0
    c->cur = 0;
    if (cudaGraphLaunch(c->gexec[q], c->stream) != cudaSuccess) {
        cudaGetLastError();
        c->graph_failed = true;
        return false;
    }
    loop_settle(c, false);
    c->launches += 1 + n;                      // begin and steps; the passes' chains are counted on the device
    return true;
}

int forces_blocks(const kg_ctx *c, int melt) { return nblk(c->sim.melt[melt].M, 128); }

void forces_eval(kg_ctx *c, int melt, long long step, double *F_dev, double *part_dev, int nb)
{
    const MeltDev &md = c->sim.melt[melt];
    ++c->launches;
    if (c->precision == KG_MIXED) {
        GeoMixed g{c->pg[c->cur], c->shtab};
        k_forces<GeoMixed><<<nb, 128, 0, c->stream>>>(c->d_sim, c->d_stage, g, c->u, md.off, md.off + md.M,
                                                     c->nl, c->nn, c->slot_of, c->bp, F_dev, part_dev, c->flags, step);
    } else {
        GeoF64 g{c->pos64[c->cur], 0.0, 0.0, {}};
        k_forces<GeoF64><<<nb, 128, 0, c->stream>>>(c->d_sim, c->d_stage, g, c->u, md.off, md.off + md.M,
                                                   c->nl, c->nn, c->slot_of, c->bp, F_dev, part_dev, c->flags, step);
    }
}

}  // namespace kg
