// kg_ppa.cu -- primitive-path analysis (PPA) of one melt and the entanglement
// length of Eq. 22 (Sec. III).  The paper measures N_e by the PPA of Everaers
// et al. (Science 303, 823 (2004)) without restating it; the form taken here:
//   * both end monomers of every chain stay fixed;
//   * the non-bonded interaction, the n = 12 member of Eq. 5 (LJ 12-6
//     truncated and shifted at 2^(1/6)), acts only between monomers of
//     different chains; inside a chain it is off, 1-2 bonded pairs included,
//     so a bond keeps its FENE part alone (Eq. 10 without U_MLJ);
//   * no bending energy (Eq. 4 off);
//   * the energy is minimised by the path's integrator at T = 0, Langevin
//     velocity Verlet with zero noise (damped dynamics), from rest.
// It runs on a copy of the melt and leaves the simulation state untouched.
//
// Storage.  The copy lives in cell order: every list build bins the monomers
// on a grid of n_c^3 cells of side h >= r_c + skin (n_c >= 3), sorts them by
// cell (a counting sort, each cell's run ordered by the previous storage index,
// so the order is deterministic) and moves every per-monomer array into that
// order, double-buffered with the buffer in use named by flag word 3.  A
// cell's monomers are then one contiguous run of storage indices, the 32
// monomers of a warp sit in a few neighbouring cells, and the candidate
// loads of the build and the neighbour gathers of the force kernel stay in
// L1 and L2.  Bonds reach their partners through a partner-index array
// refreshed at each build; results return to slot order (chain-major, s = c N
// + i) at the end.
//
// Neighbours: a Verlet list of interchain pairs within r_c + skin, entries
// j | q << IDX_BITS (j a storage index, q the stencil cell, which fixes the
// periodic image), column-major (entry k of monomer p at k M + p, so the loads
// of entry k by a warp are one coalesced row), rebuilt whenever a monomer has
// moved more than skin / 2 since the last build (flag word 1).  Candidates are
// tested in binary32 on the monomers' offsets from their cells' corners, with
// a margin that keeps every pair within r_c + skin: the list only has to
// contain the pairs, so its edge need not be exact.
//
// A step is the force at the present positions, the kick that ends the
// previous velocity Verlet step and the drift that begins the next (no kick in
// the first, no drift in the last of the n_iter + 1).  They run as the captured
// step loop of the MD path (kg_md.cu): passes of the list build, which returns
// at once without a request, and PPA_PASS steps, those after a request left to
// the next pass.  A contraction rebuilds its list every few steps: 200 steps
// of 200,000 monomers with 51 builds take 6.8 ms, and took 11.3 with drift and force apart
// and a conditional node per step.
//
// Two force kernels.  Binary64 (KG_FP64): minimum-image distances and forces
// in binary64, the same update order as the definition.  Mixed (KG_MIXED), the
// GB300 path, whose binary64 rate is a small fraction of its binary32 rate:
// the pair vector is (o_j + d_j) - (o_p + d_p) + q h in binary32, o the build
// offset and d the displacement since the build, so every term is small and
// the vector is good to ~1e-7 sigma.  The binary64 position is touched only
// at a build: between builds a monomer's position is its binary64 build
// position plus d, and every step runs in binary32 (a bond vector is its
// build value, a binary64 difference rounded to binary32, plus the
// difference of the two displacements); the build folds d into the binary64
// position.  Force, kick and drift are one kernel there: records and
// displacements alternate between two buffers from step to step, since
// neighbours read them while their owner moves on.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <vector>

#include "kg_host.h"

namespace kg {

// kg_md.cu: exclusive scan of the cell counts
__global__ void k_scan1(const int *__restrict__ in, int *__restrict__ out, int *__restrict__ bsum, int n,
                        const unsigned *__restrict__ flags);
__global__ void k_scan2(int *__restrict__ out, const int *__restrict__ bsum, int n, int nblk,
                        const unsigned *__restrict__ flags);

namespace {

constexpr double PPA_RC = 1.122462048309373;   // 2^(1/6)
constexpr int PPA_MAXNB = 128;                  // list entries per monomer (overflow: capacity error)
constexpr int PPA_CELL_CAP = 1024;              // monomers per cell the build accepts
constexpr int PPA_PASS = 6;                     // steps per pass of the captured loop (even; a build every 4 to 7 steps)
constexpr int PPA_DIRECT_PASS = 2;              // the same without a graph
constexpr long long PPA_GRAPH_MIN = 16;         // steps that are worth a capture (~0.2 ms; more than one pass)
constexpr int PPA_BLOCK = 128;
constexpr int PPA_ILP = 4;                      // list entries in flight per thread (mixed force)
constexpr unsigned FIXED_BIT = 0x80000000u;     // record word w: chain index | FIXED_BIT at a chain end

struct PpaArgs {
    int M, N, nc, ncell;
    double L, invL, h, invh;     // box, 1/L, cell side and its inverse
    float hf, rl2f, rc2f;        // binary32 cell side, list radius^2 with margin, r_c^2
    double half_skin2;           // (skin / 2)^2
    double dt, gamma, k, R0sq;
    float dtf, gammaf, kf, invR0sqf, half_skin2f;
    long long n_iter;
    // per-monomer state in storage order, moved from buffer to buffer by a build; buffer flags[3] in use
    double *x0, *x1;             // (3, M) positions (mixed: positions at the last build)
    double *v0, *v1;             // (3, M) velocities, binary64 mode
    float *u0, *u1;              // (3, M) velocities, mixed mode
    int *slot0, *slot1;          // storage index -> slot
    // single-buffered, rewritten at each build (storage order of the new buffer)
    double *xb;                  // positions at the build (binary64 mode)
    double *F;                   // (3, M) forces of the step, binary64 mode
    float *G;                    // (3, M) forces of the last step, mixed mode
    float4 *rec;                 // build offset + (chain | FIXED_BIT)
    float4 *pg[2], *dl[2];       // mixed: offset + d; d (buffers alternate between steps)
    float4 *off;                 // bin output in the old order: offset + cell index
    float4 *bvec;                // mixed: bond vector to the next monomer at the build
    int2 *bp;                    // storage indices of the bonded partners (-1 past an end)
    int *pos_of;                 // slot -> storage index
    int *cellof;                 // packed cell coordinates of each storage index
    int *rank, *count, *start, *list, *nn;
    unsigned *nl;                // entries j | q << IDX_BITS, column-major
    unsigned *flags;             // [0] error bits, [1] rebuild request, [2] builds, [3] buffer in use, [6] launches
    LoopDev *loop;
    long long *steps;            // steps completed before the present pass
};

__device__ __forceinline__ int cur_buf(const PpaArgs &a) { return (int)(a.flags[3] & 1u); }
// the buffer of the steps of a pass: a build requested before it has moved the arrays to the other one
__device__ __forceinline__ int step_buf(const PpaArgs &a) { return (int)((a.flags[3] ^ a.flags[1]) & 1u); }
__device__ __forceinline__ bool build_requested(const PpaArgs &a) { return a.flags[1] && !a.flags[0]; }

__device__ __forceinline__ double min_image(double d, const PpaArgs &a)
{
    return __dsub_rn(d, __dmul_rn(a.L, rint(__dmul_rn(d, a.invL))));
}

// step_off (kg_internal.cuh), one thread's answer for the block
__device__ __forceinline__ bool block_off(const PpaArgs &a, int k)
{
    __shared__ unsigned off;
    if (threadIdx.x == 0) off = step_off(a.flags, a.loop, k);
    __syncthreads();
    return off != 0u;
}

__device__ __forceinline__ bool is_fixed(const float4 &r) { return (__float_as_uint(r.w) & FIXED_BIT) != 0u; }

// ---- one step: force and kick, drift ----

// binary64: first half kick and drift of the mobile monomers:
// v <- v + (dt/2) F; x <- x + dt v; request a rebuild past skin / 2
__global__ void __launch_bounds__(PPA_BLOCK) k_ppa_drift_f64(PpaArgs a, int k)
{
    if (block_off(a, k) || *a.steps + k == a.n_iter) return;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.M || is_fixed(a.rec[p])) return;
    const int cb = step_buf(a);
    double *x = cb ? a.x1 : a.x0, *v = cb ? a.v1 : a.v0;
    const double hdt = 0.5 * a.dt;
    double dr2 = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const size_t o = (size_t)d * a.M + p;
        const double vh = __dadd_rn(v[o], __dmul_rn(hdt, a.F[o]));
        const double xn = __dadd_rn(x[o], __dmul_rn(a.dt, vh));
        v[o] = vh;
        x[o] = xn;
        const double e = xn - a.xb[o];
        dr2 += e * e;
    }
    if (!(dr2 <= a.half_skin2)) {
        if (!isfinite(dr2)) atomicOr(a.flags, ERR_NONFINITE);
        atomicOr(&a.loop->req, 1u << k);
    }
}

// build 1: cell of each monomer (current order) from its wrapped position,
// its offset from the cell's corner and its rank in the cell; mixed: the
// displacement d is folded into the binary64 position here, each thread on
// its own monomer (the permutation then reads positions only)
__global__ void __launch_bounds__(256) k_ppa_bin(PpaArgs a)
{
    if (!build_requested(a)) return;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.M) return;
    double *x = cur_buf(a) ? a.x1 : a.x0;
    const float4 dp = a.u0 ? a.dl[a.loop->src][p] : make_float4(0.f, 0.f, 0.f, 0.f);
    const float dd[3] = {dp.x, dp.y, dp.z};
    int cc[3];
    float o[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        double xd = x[(size_t)d * a.M + p];
        if (a.u0) {                                    // mixed: fold d into the binary64 position
            xd += f32_to_f64(dd[d]);
            x[(size_t)d * a.M + p] = xd;
        }
        cc[d] = cell_of(xd, a.h, a.invh, a.nc, o[d]);
    }
    const int c = (cc[2] * a.nc + cc[1]) * a.nc + cc[0];
    a.off[p] = make_float4(o[0], o[1], o[2], __int_as_float(c));
    // one atomic per cell and warp: neighbours in storage order share cells
    const unsigned act = __activemask(), grp = __match_any_sync(act, c);
    const int lane = threadIdx.x & 31, leader = __ffs(grp) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(a.count + c, __popc(grp));
    base = __shfl_sync(grp, base, leader);
    a.rank[p] = base + __popc(grp & ((1u << lane) - 1u));
}

// build 2: the current storage indices by cell, in no fixed order within one;
// clear the counts for the next build
__global__ void __launch_bounds__(256) k_ppa_scatter(PpaArgs a)
{
    if (!build_requested(a)) return;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    for (int c = p; c < a.ncell; c += gridDim.x * blockDim.x) {
        if (a.count[c] > PPA_CELL_CAP) atomicOr(a.flags, ERR_NL_CAPACITY);
        a.count[c] = 0;
    }
    if (p >= a.M) return;
    a.list[a.start[__float_as_int(a.off[p].w)] + a.rank[p]] = p;
}

// build 3: move every per-monomer array into cell order (the other buffer),
// a cell's run ordered by present storage index (deterministic): the new index
// is the cell's start plus the number of its members with a lower one; the
// records, displacement, build positions and slot -> storage map
__global__ void __launch_bounds__(256) k_ppa_permute(PpaArgs a)
{
    if (!build_requested(a)) return;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= a.M) return;
    const int cb = cur_buf(a);
    const int p = a.list[t];
    const size_t M = a.M;
    const float4 o = a.off[p];
    const int c = __float_as_int(o.w);
    const int b0 = a.start[c], b1 = a.start[c + 1];
    int q = b0;
    for (int k = b0; k < b1; ++k) q += a.list[k] < p;
    const double *xs = cb ? a.x1 : a.x0;
    double *xd = cb ? a.x0 : a.x1;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const double xv = xs[d * M + p];
        xd[d * M + q] = xv;
        if (a.xb) a.xb[d * M + q] = xv;
    }
    if (a.u0) {
        const float *us = cb ? a.u1 : a.u0;
        float *ud = cb ? a.u0 : a.u1;
#pragma unroll
        for (int d = 0; d < 3; ++d) ud[d * M + q] = us[d * M + p];
    } else {
        const double *vs = cb ? a.v1 : a.v0;
        double *vd = cb ? a.v0 : a.v1;
#pragma unroll
        for (int d = 0; d < 3; ++d) vd[d * M + q] = vs[d * M + p];
    }
    const int s = (cb ? a.slot1 : a.slot0)[p];
    (cb ? a.slot0 : a.slot1)[q] = s;
    a.pos_of[s] = q;
    const int i = s % a.N;
    const unsigned w = (unsigned)(s / a.N) | ((i == 0 || i == a.N - 1) ? FIXED_BIT : 0u);
    const float4 r = make_float4(o.x, o.y, o.z, __uint_as_float(w));
    a.rec[q] = r;
    if (a.u0) {
        a.pg[0][q] = r;
        a.dl[0][q] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    a.cellof[q] = (int)pack_code(c % a.nc, (c / a.nc) % a.nc, c / (a.nc * a.nc));
}

// storage indices of monomer p's bonded partners; mixed: the bond vector to
// the next monomer (binary64 difference rounded to binary32); cb: the buffer
// that the permutation wrote
__device__ __forceinline__ void partners_one(const PpaArgs &a, int p, int cb)
{
    const int s = (cb ? a.slot1 : a.slot0)[p];
    const int i = s % a.N;
    const int2 b = make_int2(i > 0 ? a.pos_of[s - 1] : -1, i < a.N - 1 ? a.pos_of[s + 1] : -1);
    a.bp[p] = b;
    if (a.bvec && b.y >= 0) {
        const double *x = cb ? a.x1 : a.x0;
        const size_t M = a.M;
        a.bvec[p] = make_float4((float)(x[b.y] - x[p]), (float)(x[M + b.y] - x[M + p]),
                                (float)(x[2 * M + b.y] - x[2 * M + p]), 0.f);
    }
}

// build 4: bonded partners and the interchain Verlet list of monomer p from
// the binary32 build offsets: every t of another chain in the 27 cells around
// p whose vector o_t - o_p + q h is shorter than r_c + skin (plus a margin
// above the offsets' rounding).  The three cells of a row in x are walked as
// one run, four candidates in flight: the lanes of a warp diverge at the ends
// of 9 runs of ~12 instead of 27 of ~4.  The thread of monomer 0 counts the
// build; the loop's end kernel makes the new buffer the one in use.
__global__ void __launch_bounds__(PPA_BLOCK) k_ppa_nlist(PpaArgs a)
{
    if (!build_requested(a)) return;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.M) return;
    if (p == 0) a.flags[2] += 1u;
    partners_one(a, p, cur_buf(a) ^ 1);
    const float4 rp = a.rec[p];
    const unsigned chain = __float_as_uint(rp.w) & ~FIXED_BIT;
    const unsigned code = (unsigned)a.cellof[p];
    const int cx = (int)(code & CODE_MASK), cy = (int)((code >> CODE_BITS) & CODE_MASK),
              cz = (int)(code >> (2 * CODE_BITS));
    const int nc = a.nc;
    auto wrap = [nc](int v) { return v < 0 ? v + nc : (v >= nc ? v - nc : v); };
    const int xl = wrap(cx - 1), xr = wrap(cx + 1);
    int n = 0;
    for (int r = 0; r < 9; ++r) {
        const int dz = r / 3 - 1, dy = r % 3 - 1;
        const int zy = (wrap(cz + dz) * nc + wrap(cy + dy)) * nc;
        const float sy = (float)dy * a.hf - rp.y, sz = (float)dz * a.hf - rp.z;
        // the row's cells left, centre, right as one run of candidates
        const int b0 = __ldg(a.start + zy + xl), b1 = __ldg(a.start + zy + cx), b2 = __ldg(a.start + zy + xr);
        const int n0 = __ldg(a.start + zy + xl + 1) - b0;
        const int n1 = n0 + __ldg(a.start + zy + cx + 1) - b1;
        const int n2 = n1 + __ldg(a.start + zy + xr + 1) - b2;
        for (int k = 0; k < n2; k += 4) {
            float4 rj[4];
            int j[4];
            int dx[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int t = min(k + i, n2 - 1);
                j[i] = t < n0 ? b0 + t : t < n1 ? b1 + (t - n0) : b2 + (t - n1);
                dx[i] = t < n0 ? -1 : t < n1 ? 0 : 1;
                rj[i] = __ldg(a.rec + j[i]);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float sx = (float)dx[i] * a.hf - rp.x;
                const float ex = rj[i].x + sx, ey = rj[i].y + sy, ez = rj[i].z + sz;
                if (k + i < n2 && (__float_as_uint(rj[i].w) & ~FIXED_BIT) != chain &&
                    ex * ex + ey * ey + ez * ez < a.rl2f) {
                    if (n < PPA_MAXNB) a.nl[(size_t)n * a.M + p] = (unsigned)j[i] | ((unsigned)(3 * r + 1 + dx[i]) << IDX_BITS);
                    ++n;
                }
            }
        }
    }
    if (n > PPA_MAXNB) {
        atomicOr(a.flags, ERR_NL_CAPACITY);
        n = PPA_MAXNB;
    }
    a.nn[p] = n;
}

// binary64 force: minimum-image pair vectors, LJ 12-6 between chains, FENE
// bonds; F <- F_c(x) - gamma v; v <- v + half dt F (half = 0 for the first force)
__global__ void __launch_bounds__(PPA_BLOCK) k_ppa_force_f64(PpaArgs a, int k)
{
    if (block_off(a, k)) return;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.M || is_fixed(a.rec[p])) return;
    const int cb = step_buf(a);
    const double *x = cb ? a.x1 : a.x0;
    double *v = cb ? a.v1 : a.v0, *F = a.F;
    const size_t M = a.M;
    const double xs = x[p], ys = x[M + p], zs = x[2 * M + p];
    double fx = 0.0, fy = 0.0, fz = 0.0;
    const int n = a.nn[p];
    const double rc2 = PPA_RC * PPA_RC;
    for (int i = 0; i < n; ++i) {
        const int j = (int)(a.nl[(size_t)i * M + p] & IDX_MASK);
        const double ex = min_image(__dsub_rn(x[j], xs), a);
        const double ey = min_image(__dsub_rn(x[M + j], ys), a);
        const double ez = min_image(__dsub_rn(x[2 * M + j], zs), a);
        const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez));
        if (r2 < rc2) {
            const double ir2 = 1.0 / r2;
            const double ir6 = ir2 * ir2 * ir2;
            const double g = (48.0 * ir6 * ir6 - 24.0 * ir6) * ir2;   // -U'(r)/r, U = 4(r^-12 - r^-6) + 1
            fx -= g * ex;
            fy -= g * ey;
            fz -= g * ez;
        }
    }
    const int2 b = a.bp[p];
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const int t = side ? b.y : b.x;
        const double bx = __dsub_rn(x[t], xs), by = __dsub_rn(x[M + t], ys), bz = __dsub_rn(x[2 * M + t], zs);
        const double q = __dadd_rn(__dadd_rn(__dmul_rn(bx, bx), __dmul_rn(by, by)), __dmul_rn(bz, bz)) / a.R0sq;
        if (!(q < 1.0)) {
            atomicOr(a.flags, ERR_OVERSTRETCH);
            continue;
        }
        const double gb = a.k / (1.0 - q);
        fx += gb * bx;
        fy += gb * by;
        fz += gb * bz;
    }
    const double hdt = (*a.steps + k ? 0.5 : 0.0) * a.dt;
    const double f[3] = {fx, fy, fz};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const size_t o = (size_t)d * M + p;
        const double vh = v[o];
        const double Ft = __dsub_rn(f[d], __dmul_rn(a.gamma, vh));
        F[o] = Ft;
        v[o] = __dadd_rn(vh, __dmul_rn(hdt, Ft));
    }
}

// One step of the mixed path, all binary32.  Pair vectors from the gather
// records, LJ 12-6; bond vectors from the build's bond vectors and the
// displacements; FENE, friction, the kick, and the next step's half kick and
// drift into the displacement since the build; a build request past skin / 2.
// Bound by the latency of the list and record gathers: PPA_ILP entries are in
// flight per thread, and the image shifts come from a word table in shared
// memory (27 words in 27 banks).
__global__ void __launch_bounds__(PPA_BLOCK) k_ppa_step_mixed(PpaArgs a, int k)
{
    __shared__ float sh[96];
    for (int q = threadIdx.x; q < 96; q += PPA_BLOCK) {
        const int i = q & 31, c = i < 27 ? (q < 32 ? i % 3 : q < 64 ? (i / 3) % 3 : i / 9) - 1 : 0;
        sh[q] = (float)c * a.hf;
    }
    if (block_off(a, k)) return;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.M) return;
    const float4 *__restrict__ pg = a.pg[k & 1], *__restrict__ dl = a.dl[k & 1];
    const long long step = *a.steps + k;
    const float4 ps = pg[p];
    if (is_fixed(ps)) {
        a.pg[~k & 1][p] = ps;
        a.dl[~k & 1][p] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    float *u = step_buf(a) ? a.u1 : a.u0;
    const size_t M = a.M;
    float fx = 0.f, fy = 0.f, fz = 0.f;
    const int n = a.nn[p];
    for (int i0 = 0; i0 < n; i0 += PPA_ILP) {
        unsigned e[PPA_ILP];
        float4 pj[PPA_ILP];
#pragma unroll
        for (int i = 0; i < PPA_ILP; ++i) e[i] = i0 + i < n ? __ldg(a.nl + (size_t)(i0 + i) * M + p) : (unsigned)p;
#pragma unroll
        for (int i = 0; i < PPA_ILP; ++i) pj[i] = __ldg(pg + (e[i] & IDX_MASK));
#pragma unroll
        for (int i = 0; i < PPA_ILP; ++i) {
            const unsigned q = e[i] >> IDX_BITS;
            const float ex = (pj[i].x - ps.x) + sh[q], ey = (pj[i].y - ps.y) + sh[32 + q],
                        ez = (pj[i].z - ps.z) + sh[64 + q];
            const float r2 = ex * ex + ey * ey + ez * ez;
            if (r2 < a.rc2f && i0 + i < n) {
                const float ir2 = __frcp_rn(r2);
                const float ir6 = ir2 * ir2 * ir2;
                const float g = (48.f * ir6 * ir6 - 24.f * ir6) * ir2;   // -U'(r)/r, U = 4(r^-12 - r^-6) + 1
                fx -= g * ex;
                fy -= g * ey;
                fz -= g * ez;
            }
        }
    }
    const int2 b = a.bp[p];
    const float4 dp = dl[p];
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const int t = side ? b.y : b.x;
        const float4 dt_ = __ldg(dl + t);
        const float4 bv = __ldg(a.bvec + (side ? p : t));
        const float sg = side ? 1.f : -1.f;             // the previous bond is -(its bond to p)
        const float bx = sg * bv.x + (dt_.x - dp.x), by = sg * bv.y + (dt_.y - dp.y),
                    bz = sg * bv.z + (dt_.z - dp.z);
        const float q = (bx * bx + by * by + bz * bz) * a.invR0sqf;
        if (!(q < 1.f)) {
            atomicOr(a.flags, ERR_OVERSTRETCH);
            continue;
        }
        const float gb = a.kf * __frcp_rn(1.f - q);
        fx += gb * bx;
        fy += gb * by;
        fz += gb * bz;
    }
    const float hdt = (step ? 0.5f : 0.f) * a.dtf, hdt2 = 0.5f * a.dtf;
    const float f[3] = {fx, fy, fz};
    const bool last = step == a.n_iter;
    float dd[3] = {dp.x, dp.y, dp.z};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const size_t o = (size_t)d * M + p;
        const float vh = u[o];
        const float Ft = f[d] - a.gammaf * vh;
        float un = vh + hdt * Ft;
        if (last) {
            a.G[o] = Ft;
        } else {
            un = un + hdt2 * Ft;
            dd[d] += a.dtf * un;
        }
        u[o] = un;
    }
    a.dl[~k & 1][p] = make_float4(dd[0], dd[1], dd[2], 0.f);
    if (last) return;
    const float4 r = a.rec[p];
    a.pg[~k & 1][p] = make_float4(r.x + dd[0], r.y + dd[1], r.z + dd[2], r.w);
    const float dr2 = dd[0] * dd[0] + dd[1] * dd[1] + dd[2] * dd[2];
    if (!(dr2 <= a.half_skin2f)) {
        if (!isfinite(dr2)) atomicOr(a.flags, ERR_NONFINITE);
        atomicOr(&a.loop->req, 1u << k);
    }
}

// ---- results in slot order ----

// one monomer back to slot order; the bits of its net force (0 at a chain end)
__device__ __forceinline__ unsigned long long unpermute_one(const PpaArgs &a, int s, double *__restrict__ xs)
{
    const int cb = cur_buf(a);
    const double *x = cb ? a.x1 : a.x0;
    const size_t M = a.M;
    const int p = a.pos_of[s];
    const float4 dp = a.u0 ? a.dl[a.loop->par][p] : make_float4(0.f, 0.f, 0.f, 0.f);
    const float dd[3] = {dp.x, dp.y, dp.z};
    double f2 = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        xs[d * M + s] = x[d * M + p] + (double)dd[d];
        const double f = a.u0 ? (double)a.G[d * M + p] : a.F[d * M + p];
        f2 += f * f;
    }
    const int i = s % a.N;
    return (i > 0 && i < a.N - 1) ? (unsigned long long)__double_as_longlong(sqrt(f2)) : 0ull;
}

// positions back to slot order; the largest net force on a mobile monomer
// (a warp maximum, then one atomic per warp) and the sum of the list lengths.
// A first build cut short (a cell over PPA_CELL_CAP: flags[2] is 0) has not
// written the index arrays, which are not cleared beforehand, and nothing has
// moved: buffer 0 holds the positions in slot order.
__global__ void __launch_bounds__(256) k_ppa_unpermute(PpaArgs a, double *__restrict__ xs,
                                                      unsigned long long *__restrict__ fmax_bits,
                                                      unsigned long long *__restrict__ nn_sum)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long fb = 0ull;                      // bits of a non-negative double order like it
    unsigned long long nb = 0ull;
    if (s < a.M && a.flags[2]) {
        fb = unpermute_one(a, s, xs);
        nb = (unsigned long long)a.nn[s];              // list lengths, storage order (any order sums)
    } else if (s < a.M) {
#pragma unroll
        for (int d = 0; d < 3; ++d) xs[(size_t)d * a.M + s] = a.x0[(size_t)d * a.M + s];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long t = __shfl_down_sync(0xffffffffu, fb, o);
        fb = t > fb ? t : fb;
        nb += __shfl_down_sync(0xffffffffu, nb, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (fb) atomicMax(fmax_bits, fb);
        atomicAdd(nn_sum, nb);
    }
}

// contour length of every chain from slot-order positions: one warp per
// chain, lane l sums bonds l, l + 32, ..., then a fixed-order shuffle tree
__global__ void __launch_bounds__(256) k_ppa_lengths(const double *__restrict__ x, int M, int N,
                                                    double *__restrict__ lpp)
{
    const int c = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (c >= M / N) return;
    double sum = 0.0;
    for (int i = lane; i + 1 < N; i += 32) {
        const size_t s = (size_t)c * N + i;
        const double bx = __dsub_rn(x[s + 1], x[s]);
        const double by = __dsub_rn(x[M + s + 1], x[M + s]);
        const double bz = __dsub_rn(x[2 * (size_t)M + s + 1], x[2 * (size_t)M + s]);
        sum += sqrt(__dadd_rn(__dadd_rn(__dmul_rn(bx, bx), __dmul_rn(by, by)), __dmul_rn(bz, bz)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
    if (lane == 0) lpp[c] = sum;
}

__global__ void k_ppa_iota(int *__restrict__ a, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) a[i] = i;
}

inline int nblk(long long n, int b) { return (int)((n + b - 1) / b); }

// ends a pass: the buffer that a build wrote becomes the one in use
__global__ void k_ppa_end(PpaArgs a, int len, cudaGraphConditionalHandle h, int in_graph)
{
    a.flags[3] ^= a.flags[1];
    const bool more = loop_finish(a.loop, len, a.steps, a.flags);
    if (in_graph) cudaGraphSetConditional(h, more ? 1u : 0u);
}

// one pass: the list build (each kernel returns at once unless a build is
// requested), `len` steps, the end kernel (h: the loop's condition in a graph)
void enqueue_pass(const PpaArgs &a, cudaStream_t st, int *bsum, bool mixed, int len, cudaGraphConditionalHandle h,
                  bool in_graph)
{
    const int nbs = nblk(a.ncell, 1024), nbm = nblk(a.M, PPA_BLOCK);
    k_ppa_bin<<<nblk(a.M, 256), 256, 0, st>>>(a);
    k_scan1<<<nbs, 1024, 0, st>>>(a.count, a.start, bsum, a.ncell, a.flags);
    k_scan2<<<nbs, 1024, 0, st>>>(a.start, bsum, a.ncell, nbs, a.flags);
    k_ppa_scatter<<<nblk(a.M, 256), 256, 0, st>>>(a);
    k_ppa_permute<<<nblk(a.M, 256), 256, 0, st>>>(a);
    k_ppa_nlist<<<nbm, PPA_BLOCK, 0, st>>>(a);
    for (int k = 0; k < len; ++k) {
        if (mixed) {
            k_ppa_step_mixed<<<nbm, PPA_BLOCK, 0, st>>>(a, k);
        } else {
            k_ppa_force_f64<<<nbm, PPA_BLOCK, 0, st>>>(a, k);
            k_ppa_drift_f64<<<nbm, PPA_BLOCK, 0, st>>>(a, k);
        }
    }
    k_ppa_end<<<1, 1, 0, st>>>(a, len, h, in_graph);
}

// Eq. 22's left-hand side (2 x + exp(-2 x) - 1) / (2 x^2); a series below
// x = 1e-3, where the closed form cancels
double eq22_lhs(double x)
{
    if (x < 1e-3) return 1.0 - 2.0 * x / 3.0 + x * x / 3.0 - 2.0 * x * x * x / 15.0;
    return (2.0 * x + std::expm1(-2.0 * x)) / (2.0 * x * x);
}

}  // namespace
}  // namespace kg

using namespace kg;

extern "C" {

kg_status kg_primitive_path(kg_ctx *c, int melt, const kg_ppa_params *pp, double *lpp, double *x_out,
                            kg_ppa_result *res)
{
    if (!c || !pp || melt < 0 || melt >= c->sim.n_melts) return KG_ERR_INVALID_ARG;
    if (!(pp->dt > 0.0) || !(pp->gamma >= 0.0) || !(pp->skin > 0.0) || pp->n_iter < 0) return KG_ERR_INVALID_ARG;
    if (pp->precision != KG_FP64 && pp->precision != KG_MIXED) return KG_ERR_INVALID_ARG;
    if (cudaSetDevice(c->device) != cudaSuccess) return KG_ERR_CUDA;
    if (c->latched != KG_OK) return KG_ERR_STATE;
    const MeltDev &md = c->sim.melt[melt];
    const double rl = PPA_RC + pp->skin;
    const int nc = (int)std::floor(md.L / rl);
    if (nc < 3 || nc > 1024) return KG_ERR_INVALID_ARG;     // 27 distinct stencil cells; bounded grid
    const bool mixed = pp->precision == KG_MIXED;
    const double k = pp->k_fene > 0.0 ? pp->k_fene : kg_kn(12.0, c->p.R0, c->p.l0);
    const int M = md.M, N = md.N, n_ch = md.n_ch;

    PpaArgs a{};
    a.M = M;
    a.N = N;
    a.nc = nc;
    a.ncell = nc * nc * nc;
    a.L = md.L;
    a.invL = 1.0 / md.L;
    a.h = md.L / nc;
    a.invh = nc / md.L;
    a.hf = (float)a.h;
    a.rl2f = (float)(rl * rl) + 1e-4f;          // margin >> the binary32 error of the offsets
    a.rc2f = (float)(PPA_RC * PPA_RC);
    a.half_skin2 = 0.25 * pp->skin * pp->skin;
    a.dt = pp->dt;
    a.gamma = pp->gamma;
    a.k = k;
    a.R0sq = c->p.R0 * c->p.R0;
    a.dtf = (float)pp->dt;
    a.gammaf = (float)pp->gamma;
    a.kf = (float)k;
    a.invR0sqf = (float)(1.0 / a.R0sq);
    a.half_skin2f = (float)a.half_skin2;
    a.n_iter = pp->n_iter;

    const size_t m3 = 3 * (size_t)M;
    const int nbs = nblk(a.ncell, 1024);
    // one allocation for all arrays: those that start at zero in front, cleared
    // together (26 allocations and clears took ~0.2 ms before the first kernel)
    struct Part {
        void *p;                                         // the pointer to set
        size_t bytes;
    };
    std::vector<Part> zeroed, plain;
    auto get = [](std::vector<Part> &l, auto *&p, size_t n) { l.push_back({&p, (sizeof(*p) * n + 255) & ~(size_t)255}); };
    int *bsum;
    double *d_xs, *d_lpp;
    unsigned long long *d_fmax;                          // max |F|, sum nn
    get(plain, a.x0, m3);
    get(plain, a.x1, m3);
    if (mixed) {
        get(zeroed, a.u0, m3);
        get(plain, a.u1, m3);
        get(plain, a.G, m3);
        get(plain, a.bvec, M);
        get(zeroed, a.dl[0], M);                         // the first build folds it in
        get(plain, a.dl[1], M);
        for (int b = 0; b < 2; ++b) get(plain, a.pg[b], M);
    } else {
        get(zeroed, a.v0, m3);
        get(plain, a.v1, m3);
        get(plain, a.F, m3);
        get(plain, a.xb, m3);
    }
    get(plain, a.slot0, M);
    get(plain, a.slot1, M);
    get(plain, a.rec, M);
    get(plain, a.off, M);
    get(plain, a.bp, M);
    get(plain, a.pos_of, M);
    get(plain, a.cellof, M);
    get(plain, a.rank, M);
    get(zeroed, a.count, (size_t)a.ncell + 1);
    get(plain, a.start, (size_t)a.ncell + 1);
    get(plain, a.list, M);
    get(plain, a.nl, (size_t)PPA_MAXNB * M);
    get(plain, a.nn, M);
    get(zeroed, a.flags, 8);
    get(zeroed, a.loop, 1);
    get(zeroed, a.steps, 1);
    get(plain, bsum, nbs);
    get(plain, d_xs, m3);
    get(plain, d_lpp, n_ch);
    get(zeroed, d_fmax, 2);
    size_t clear = 0, bytes = 0;
    for (const Part &q : zeroed) clear += q.bytes;
    for (const Part &q : plain) bytes += q.bytes;
    char *const pool = (char *)dev_alloc(c, clear + bytes, clear);
    if (!pool) return KG_ERR_OOM;
    size_t at = 0;
    for (const std::vector<Part> *l : {&zeroed, &plain})
        for (const Part &q : *l) {
            char *const here = pool + at;
            std::memcpy(q.p, &here, sizeof(here));
            at += q.bytes;
        }
    cudaStream_t gs = nullptr;
    cudaGraphExec_t gexec = nullptr;
    auto done = [&](kg_status r) {
        if (gexec) cudaGraphExecDestroy(gexec);
        if (gs) cudaStreamDestroy(gs);
        cudaStreamSynchronize(c->stream);
        dev_free(c, pool);
        return r;
    };

    cudaStream_t st = c->stream;
    kg::to_slots(c, melt, c->x, a.x0, 3);              // (3, M) slot order, unwrapped; buffer 0
    k_ppa_iota<<<nblk(M, 256), 256, 0, st>>>(a.slot0, M);
    static const unsigned one = 1u;
    if (cudaMemcpyAsync(a.flags + 1, &one, sizeof(unsigned), cudaMemcpyHostToDevice, st) != cudaSuccess)
        return done(KG_ERR_CUDA);
    // the build into cell order, then n_iter + 1 steps from rest
    const long long steps = pp->n_iter + 1;
    const int len = steps >= PPA_GRAPH_MIN ? PPA_PASS : PPA_DIRECT_PASS;
    loop_begin(st, a.loop, steps, len);
    if (len == PPA_PASS)                               // its work covers the capture's host time
        enqueue_pass(a, st, bsum, mixed, len, cudaGraphConditionalHandle{}, false);
    if (len == PPA_PASS && cudaStreamCreateWithFlags(&gs, cudaStreamNonBlocking) == cudaSuccess &&
        capture_loop(gs, &gexec, [&](cudaGraphConditionalHandle h) { enqueue_pass(a, gs, bsum, mixed, len, h, true); })) {
        if (cudaGraphLaunch(gexec, st) != cudaSuccess) return done(KG_ERR_CUDA);
    } else {                                           // a pass does one step at least; none is left for the last ones
        for (long long i = 0; i < steps; ++i) enqueue_pass(a, st, bsum, mixed, len, cudaGraphConditionalHandle{}, false);
    }
    k_ppa_unpermute<<<nblk(M, 256), 256, 0, st>>>(a, d_xs, d_fmax, d_fmax + 1);
    k_ppa_lengths<<<nblk(32LL * n_ch, 256), 256, 0, st>>>(d_xs, M, N, d_lpp);
    if (cudaGetLastError() != cudaSuccess) return done(KG_ERR_CUDA);

    std::vector<double> h_lpp((size_t)n_ch);
    unsigned h_flags[8] = {};
    unsigned long long h_fmax[2] = {0, 0};
    if (cudaMemcpyAsync(h_lpp.data(), d_lpp, sizeof(double) * n_ch, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemcpyAsync(h_flags, a.flags, sizeof(h_flags), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemcpyAsync(h_fmax, d_fmax, sizeof(h_fmax), cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return done(KG_ERR_CUDA);
    kg::follow_default_for(c, x_out);
    if (x_out && cudaMemcpyAsync(x_out, d_xs, sizeof(double) * m3, cudaMemcpyDefault, st) != cudaSuccess)
        return done(KG_ERR_CUDA);
    if (cudaStreamSynchronize(st) != cudaSuccess) return done(KG_ERR_CUDA);
    c->launches += 5 + (mixed ? 1 : 2) * steps + (long long)h_flags[6];   // the passes' other kernels: counted there
    const unsigned e = h_flags[0];
    if (e & ERR_OVERSTRETCH) return done(KG_ERR_BOND_OVERSTRETCH);
    if (e & ERR_NONFINITE) return done(KG_ERR_NONFINITE);
    if (e & ERR_NL_CAPACITY) return done(KG_ERR_CAPACITY);
    if (lpp)
        for (int i = 0; i < n_ch; ++i) lpp[i] = h_lpp[(size_t)i];
    if (res) {
        double sum = 0.0;
        for (double v : h_lpp) sum += v;               // chain order
        res->lpp_mean = sum / (double)n_ch;
        std::memcpy(&res->fmax, &h_fmax[0], sizeof(double));
        res->builds = (long long)h_flags[2];
        res->mean_neighbours = (double)h_fmax[1] / (double)M;
    }
    return done(KG_OK);
}

kg_status kg_entanglement_length(double lpp_mean, int chain_len, double l0, double l_k, double *n_ek, double *n_e)
{
    if (!n_ek || chain_len < 2 || !(l0 > 0.0) || !(lpp_mean > 0.0)) return KG_ERR_INVALID_ARG;
    const double r = lpp_mean / ((double)(chain_len - 1) * l0);
    const double y = r * r;
    if (!(y > 0.0 && y < 1.0)) return KG_ERR_INVALID_ARG;
    // the left-hand side falls monotonically from 1 to 0: bisection in log x
    double lo = -40.0, hi = 40.0;
    for (int it = 0; it < 200 && hi - lo > 1e-15; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (eq22_lhs(std::exp(mid)) > y) lo = mid;
        else hi = mid;
    }
    *n_ek = std::exp(0.5 * (lo + hi));
    if (n_e) {
        if (!(l_k > 0.0)) return KG_ERR_INVALID_ARG;
        *n_e = *n_ek * l_k / l0;
    }
    return KG_OK;
}

}  // extern "C"
