// kg_rebuild.cuh -- per-item work of the Verlet-list rebuild chain (binning,
// scatter into cell order, in-cell rank, list build), shared by the
// standalone rebuild kernels and the resident kernels, so both run the
// same arithmetic.
#pragma once
#include <cuda_runtime.h>

#include "kg_internal.cuh"

namespace kg {

// finite binary64 value (exponent field not all ones), tested on the bits
__device__ __forceinline__ bool finite64(double v)
{
    return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000;
}

// Monomer s: its position (mixed: build position + displacement dread since the
// build, folded into the binary64 arrays), its Verlet-grid cell and offset
// from the cell corner (the build record), the gather records reset to the
// record, and its rank within its cell (atomic count, aggregated per warp).
// Returns error bits.
__device__ __forceinline__ unsigned bin_md_one(const SimDev &S, int s, double *__restrict__ x,
                                               double *__restrict__ xb64, float4 *__restrict__ recb,
                                               const float4 *dread, float4 *dcur, float4 *__restrict__ pgcur,
                                               double4_32a *__restrict__ pcur, double4_32a *__restrict__ xb,
                                               int *__restrict__ cellid, int *__restrict__ rank,
                                               int *__restrict__ count, const int *__restrict__ slot_of,
                                               int *cell_out = nullptr, int *rank_out = nullptr)
{
    const MeltDev &md = S.melt[melt_of(S, slot_of[s])];
    const int Mp = S.Mp;
    double xs[3];
    if (xb64) {                        // mixed: the build position plus the displacement since
        const float4 e = dread[s];
        xs[0] = __dadd_rn(xb64[s], f32_to_f64(e.x));
        xs[1] = __dadd_rn(xb64[Mp + s], f32_to_f64(e.y));
        xs[2] = __dadd_rn(xb64[2 * Mp + s], f32_to_f64(e.z));
    } else {
        xs[0] = x[s];
        xs[1] = x[Mp + s];
        xs[2] = x[2 * Mp + s];
    }
    if (!(finite64(xs[0]) && finite64(xs[1]) && finite64(xs[2]))) {   // never bin a non-finite position
        return ERR_NONFINITE;
    }
    if (xb64) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            xb64[d * Mp + s] = xs[d];
            x[d * Mp + s] = xs[d];     // the band check of the list build reads x
        }
    }
    float off[3];
    int cell[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) cell[d] = cell_of(xs[d], md.h, md.invh, md.nc, off[d]);
    const float4 rb = make_float4(off[0], off[1], off[2], __uint_as_float(pack_code(cell[0], cell[1], cell[2])));
    recb[s] = rb;
    if (dcur) dcur[s] = make_float4(0.f, 0.f, 0.f, 0.f);
    pgcur[s] = make_float4(rb.x + 0.f, rb.y + 0.f, rb.z + 0.f, rb.w);
    if (pcur) {
        const double4_32a p = make_double4_32a(xs[0], xs[1], xs[2], 0.0);
        pcur[s] = p;
        xb[s] = p;
    }
    const int c = md_cell(md, cell[0], cell[1], cell[2]);
    cellid[s] = c;
    // one atomic per cell and warp: monomers in cell order share cells with
    // their lane neighbours (the in-cell order is fixed later by the rank pass)
    const unsigned act = __activemask();
    const unsigned grp = __match_any_sync(act, c);
    const int lane = threadIdx.x & 31, leader = __ffs(grp) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(count + c, __popc(grp));
    base = __shfl_sync(grp, base, leader);
    const int rk = base + __popc(grp & ((1u << lane) - 1u));
    rank[s] = rk;
    if (cell_out) *cell_out = c;
    if (rank_out) *rank_out = rk;
    return 0;
}

// Monomer s into its cell's segment of the cell-ordered list, at its
// arrival rank (the in-cell order is fixed afterwards).
__device__ __forceinline__ void scatter_one(int s, const int *__restrict__ cellid, const int *__restrict__ rank,
                                            const int *__restrict__ start, int *__restrict__ list)
{
    list[start[cellid[s]] + rank[s]] = s;
}

// Position p of the cell-ordered list: the monomer the scatter put there
// (in atomic-arrival order within its cell, tmp) moves to its rank by
// compute index among its cell's members, with its build record (w = the
// compute index), so a cell's candidates form one contiguous run in a fixed
// order (deterministic lists).  A cell's first position clears its count for
// the next build.  True if the cell holds more than MAX_CELL_OCC monomers
// (left in arrival order: an error).
__device__ __forceinline__ bool cellrank_one(int p, const int *__restrict__ cellid, const int *__restrict__ start,
                                             const int *__restrict__ tmp, int *__restrict__ list,
                                             const float4 *__restrict__ recb, float4 *__restrict__ recs,
                                             int *__restrict__ count)
{
    const int v = tmp[p];
    const int c = cellid[v];
    const int a = start[c], b = start[c + 1];
    if (p == a) count[c] = 0;
    const bool over = b - a > MAX_CELL_OCC;
    int r = p - a;
    if (!over) {
        r = 0;
        for (int q = a; q < b; ++q) r += tmp[q] < v ? 1 : 0;
    }
    list[a + r] = v;
    const float4 rb = recb[v];
    recs[a + r] = make_float4(rb.x, rb.y, rb.z, __int_as_float(v));
    return over;
}

// ---------------------------------------------------------------------------
// Verlet list of monomer s: every t != s, not 1-2 bonded, with r^2 < (r_c +
// skin)^2.  Candidates come from the 27 cells around the cell of s; a
// candidate j of stencil cell (dx, dy, dz) lies at off_j - (off_s - (dx, dy,
// dz) h) from s with no wrap, because that cell's image sits at (c_s + d) h.
// This binary32 value decides every pair outside the band [nl_lo, nl_hi),
// which bounds its rounding error; pairs inside the band are decided by the
// binary64 distance ((dx*dx + dy*dy) + dz*dz), dx = d - L rint(d/L), exactly
// as the definition.  Each entry stores j with its stencil code q, the image
// shift of the pair until the next build.
//
// A warp walks the 27 stencil cells in lockstep (all 32 lanes must call
// nlist_one together): for cell q every lane runs the warp's largest count of
// that cell; lanes past their own count load the records that follow their
// cell (recs is padded by MAX_CELL_OCC records past the last monomer, so
// every such load is in bounds) and mask them.  The candidate loop has no
// branch but its own: the append is a predicated store, and a pair inside the binary64
// band is taken provisionally and counted; a lane with band pairs re-walks
// its row after the stencil, decides each band entry by the binary64
// distance and compacts the row in place (order kept).  The candidate's
// offsets and compute index arrive in one 16-byte load.
// ---------------------------------------------------------------------------
struct MeltNl {
    int off, cell_off, nbk, nc;
    float h, lo, hi, invL;
    double L;
};

struct NlArgs {
    const double *x;         // binary64 positions [3][Mp] (band decisions)
    const float4 *recb;      // build records of the compute order
    const float4 *recs;      // the same in cell order, w = compute index
    const int *start;        // cell starts (cell order)
    unsigned *nl;            // out: entries j | q << IDX_BITS, column-major [maxnb][Mp]
    int *nn;                 // out: list lengths
    unsigned *flags;
    const int *slot_of;
    const int4 *bp;          // chain partners (1-2 bonded: y, z)
    int M, Mp, maxnb, n_melts;
    double rl2;
    MeltNl melt[MAX_MELTS];
};

__device__ __forceinline__ void st_pred(unsigned *addr, unsigned v, bool p)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q st.global.u32 [%0], %1;\n\t}"
                 ::"l"(addr), "r"(v), "r"((unsigned)p) : "memory");
}

// the same, for memory that the code around it does not read before nl_fence():
// loads may move across it
__device__ __forceinline__ void st_pred_free(unsigned *addr, unsigned v, bool p)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q st.global.u32 [%0], %1;\n\t}"
                 ::"l"(addr), "r"(v), "r"((unsigned)p));
}

__device__ __forceinline__ void nl_fence() { asm volatile("" ::: "memory"); }

// binary32 squared distance of the build records of s (ri) and t (rj) for a
// pair in stencil cell (dx, dy, dz) of s: the same expression as the build's
__device__ __forceinline__ float nl_r2(float4 ri, float4 rj, int dx, int dy, int dz, float h)
{
    const float ox = ri.x - (float)dx * h, oy = ri.y - (float)dy * h, oz = ri.z - (float)dz * h;
    const float ex = rj.x - ox, ey = rj.y - oy, ez = rj.z - oz;
    return ex * ex + ey * ey + ez * ez;
}

// The list of monomer s (s >= M: an idle lane that takes part in the warp's
// lockstep and writes nothing); returns error bits.  READ_ONLY: what it loads is not written
// in the same launch (non-coherent loads).
template <bool READ_ONLY, typename T>
__device__ __forceinline__ T nl_ld(const T *p)
{
    if constexpr (READ_ONLY) return __ldg(p);
    else return *p;
}

template <bool READ_ONLY>
__device__ __forceinline__ unsigned nlist_one(const NlArgs &A, int s)
{
    constexpr unsigned FULL = 0xffffffffu;
    const bool live = s < A.M;
    const int sv = live ? s : A.M - 1;                       // idle lanes read valid memory, write nothing
    const int slot = nl_ld<READ_ONLY>(A.slot_of + sv);
    int m = 0;
    while (m + 1 < A.n_melts && slot >= A.melt[m + 1].off) ++m;
    const MeltNl &md = A.melt[m];
    const int4 bp = nl_ld<READ_ONLY>(A.bp + sv);                        // 1-2 bonded partners: bp.y, bp.z
    const float4 ri = nl_ld<READ_ONLY>(A.recb + sv);
    const unsigned code = __float_as_uint(ri.w);
    const int cx = (int)(code & CODE_MASK), cy = (int)((code >> CODE_BITS) & CODE_MASK);
    const int cz = (int)(code >> (2 * CODE_BITS));
    const int nc = md.nc, nbk = md.nbk;
    const float h = md.h, lo = md.lo, hi = md.hi;
    const int maxnb = A.maxnb;
    const size_t Mp = (size_t)A.Mp;
    unsigned *__restrict__ out = A.nl + (live ? s : 0);
    int cnt = 0, nband = 0;
    unsigned err = 0;
#pragma unroll 1
    for (int dz = -1; dz <= 1; ++dz) {
        int zz = cz + dz;
        zz = zz < 0 ? nc - 1 : (zz >= nc ? 0 : zz);
#pragma unroll 1
        for (int dy = -1; dy <= 1; ++dy) {
            int yy = cy + dy;
            yy = yy < 0 ? nc - 1 : (yy >= nc ? 0 : yy);
            const int rowb = md.cell_off + (((zz >> 2) * nbk + (yy >> 2)) * nbk << 6) + ((zz & 3) << 4) + ((yy & 3) << 2);
#pragma unroll
            for (int dx = -1; dx <= 1; ++dx) {
                int xx = cx + dx;
                xx = xx < 0 ? nc - 1 : (xx >= nc ? 0 : xx);
                const int cell = rowb + ((xx >> 2) << 6) + (xx & 3);
                const int k0 = nl_ld<READ_ONLY>(A.start + cell);
                int n = live ? nl_ld<READ_ONLY>(A.start + cell + 1) - k0 : 0;
                if (n > MAX_CELL_OCC) {
                    err = ERR_NL_CAPACITY;
                    n = 0;
                }
                const int nmax = __reduce_max_sync(FULL, n);
                const float ox = ri.x - (float)dx * h, oy = ri.y - (float)dy * h, oz = ri.z - (float)dz * h;
                const unsigned tag = (unsigned)((dz + 1) * 9 + (dy + 1) * 3 + (dx + 1)) << IDX_BITS;
#pragma unroll 2
                for (int j = 0; j < nmax; ++j) {
                    const float4 rj = nl_ld<READ_ONLY>(A.recs + k0 + j);
                    const int t = __float_as_int(rj.w);
                    const float ex = rj.x - ox, ey = rj.y - oy, ez = rj.z - oz;
                    const float r2 = ex * ex + ey * ey + ez * ez;
                    const bool take = (j < n) & (r2 < hi) & (t != s) & (t != bp.y) & (t != bp.z);
                    nband += (take & (r2 >= lo)) ? 1 : 0;
                    st_pred_free(out + (size_t)cnt * Mp, (unsigned)t | tag, take & (cnt < maxnb));
                    cnt += take ? 1 : 0;
                }
            }
        }
    }
    nl_fence();
    if (nband > 0 && cnt <= maxnb) {                         // rare: decide the band entries in binary64
        int w = 0;
        for (int k = 0; k < cnt; ++k) {
            const unsigned e = out[(size_t)k * Mp];
            const int t = (int)(e & IDX_MASK), q = (int)(e >> IDX_BITS);
            const float r2 = nl_r2(ri, nl_ld<READ_ONLY>(A.recb + t), q % 3 - 1, (q / 3) % 3 - 1, q / 9 - 1, h);
            const bool keep = r2 < lo || dist2_exact(A.x, A.Mp, md.L, md.invL, s, t) < A.rl2;
            if (keep) out[(size_t)(w++) * Mp] = e;
        }
        cnt = w;
    }
    if (live) {
        A.nn[s] = cnt < maxnb ? cnt : maxnb;
        if (cnt > maxnb) {
            err |= ERR_NL_CAPACITY;
            atomicMax(A.flags + 3, (unsigned)cnt);
        }
    }
    return err;
}

// r^2 - hi of candidate r seen from the shifted own offset (ox, oy, oz)
__device__ __forceinline__ float nl_v(float4 r, float ox, float oy, float oz, float hi)
{
    const float ex = r.x - ox, ey = r.y - oy, ez = r.z - oz;
    return fmaf(ez, ez, fmaf(ey, ey, fmaf(ex, ex, -hi)));
}

// After a walk that took the band pairs provisionally: those of the warp's rows
// decided in binary64, the length written; near: the smallest |v| that the
// lane's row saw, m: its melt.  Whole warps.  Returns error bits.
__device__ __forceinline__ unsigned nlist_finish(const NlArgs &A, int s, int m, bool live, float near, int cnt,
                                                 int &n_out)
{
    constexpr unsigned FULL = 0xffffffffu;
    const int maxnb = A.maxnb;
    const size_t Mp = (size_t)A.Mp;
    unsigned err = 0;
    unsigned fix = __ballot_sync(FULL, live && near < (A.melt[m].hi - A.melt[m].lo) && cnt <= maxnb);
    const int lane = threadIdx.x & 31;
    __syncwarp();
    while (fix) {
        const int src = __ffs(fix) - 1;
        fix &= fix - 1;
        const int ss = __shfl_sync(FULL, s, src), cs = __shfl_sync(FULL, cnt, src);
        const MeltNl &ms = A.melt[__shfl_sync(FULL, m, src)];
        const float4 rs = A.recb[ss];
        unsigned *row = A.nl + ss;
        int kept = 0;
        for (int k = lane; k - lane < cs; k += 32) {
            const unsigned e = k < cs ? row[(size_t)k * Mp] : (unsigned)ss;
            const int t = (int)(e & IDX_MASK), q = (int)(e >> IDX_BITS);
            const float v = nl_v(A.recb[t], rs.x - (float)(q % 3 - 1) * ms.h, rs.y - (float)((q / 3) % 3 - 1) * ms.h,
                                 rs.z - (float)(q / 9 - 1) * ms.h, ms.hi);
            const bool keep = k < cs && (v < ms.lo - ms.hi || dist2_exact(A.x, A.Mp, ms.L, ms.invL, ss, t) < A.rl2);
            const unsigned bal = __ballot_sync(FULL, keep);
            if (keep) row[(size_t)(kept + __popc(bal & ((1u << lane) - 1u))) * Mp] = e;
            kept += __popc(bal);
        }
        if (lane == src) cnt = kept;
        __syncwarp();
    }
    n_out = cnt < maxnb ? cnt : maxnb;
    if (live) {
        A.nn[s] = n_out;
        if (cnt > maxnb) {
            err |= ERR_NL_CAPACITY;
            atomicMax(A.flags + 3, (unsigned)cnt);
        }
    }
    return err;
}

// The same list by another walk, for the resident kernel, where load latency
// counts and not the work: the three cells of a stencil row have their starts
// in flight together, and a cell of up to 32 candidates takes two passes.  The
// first loads U candidates at a time and only collects the signs of v = r^2 -
// hi in a mask (one funnel shift per candidate; lanes past their own count drop
// the bits) and the smallest |v| seen; the second pops the lane's set bits, in
// candidate order, for the exclusions and the append, so no store waits
// between two candidate loads.  A pair inside the band -w <= v < 0 is taken
// provisionally; after the stencil the whole warp re-reads the row of a lane
// that may hold one (about one lane in 5000), an entry per lane, decides in
// binary64 and compacts it in order.  The kernel of larger systems keeps the
// walk above: it is bound by the L1 data pipe, and this one took 362 us
// against 336 per build of 1.6M monomers there (two candidates at a time).
// s >= M: an idle lane; n_out: the length; returns error bits.
template <int U>
__device__ __forceinline__ unsigned nlist_masked(const NlArgs &A, int s, int &n_out)
{
    static_assert(32 % U == 0, "a chunk of 32 candidates is whole groups");
    constexpr unsigned FULL = 0xffffffffu;
    const bool live = s < A.M;
    const int sv = live ? s : A.M - 1;                       // idle lanes read valid memory, write nothing
    const int slot = A.slot_of[sv];
    int m = 0;
    while (m + 1 < A.n_melts && slot >= A.melt[m + 1].off) ++m;
    const MeltNl &md = A.melt[m];
    const int4 bp = A.bp[sv];                                // 1-2 bonded partners: bp.y, bp.z
    const float4 ri = A.recb[sv];
    const unsigned code = __float_as_uint(ri.w);
    const int cx = (int)(code & CODE_MASK), cy = (int)((code >> CODE_BITS) & CODE_MASK);
    const int cz = (int)(code >> (2 * CODE_BITS));
    const int nc = md.nc, nbk = md.nbk;
    const float h = md.h, hi = md.hi;
    const int maxnb = A.maxnb;
    const size_t Mp = (size_t)A.Mp;
    unsigned *out = A.nl + (live ? s : 0);
    int cnt = 0;
    float near = 3.0e38f;                                    // smallest |v| of any candidate loaded
    unsigned err = 0;
#pragma unroll 1
    for (int dz = -1; dz <= 1; ++dz) {
        int zz = cz + dz;
        zz = zz < 0 ? nc - 1 : (zz >= nc ? 0 : zz);
#pragma unroll 1
        for (int dy = -1; dy <= 1; ++dy) {
            int yy = cy + dy;
            yy = yy < 0 ? nc - 1 : (yy >= nc ? 0 : yy);
            const int rowb = md.cell_off + (((zz >> 2) * nbk + (yy >> 2)) * nbk << 6) + ((zz & 3) << 4) + ((yy & 3) << 2);
            int k0[3], n[3];
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
                int xx = cx + dx - 1;
                xx = xx < 0 ? nc - 1 : (xx >= nc ? 0 : xx);
                const int cell = rowb + ((xx >> 2) << 6) + (xx & 3);
                k0[dx] = A.start[cell];
                n[dx] = A.start[cell + 1] - k0[dx];
            }
            const float oy = ri.y - (float)dy * h, oz = ri.z - (float)dz * h;
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
                if (n[dx] > MAX_CELL_OCC) {
                    err = ERR_NL_CAPACITY;
                    n[dx] = 0;
                }
                if (!live) n[dx] = 0;
                const int nmax = __reduce_max_sync(FULL, n[dx]);
                const float ox = ri.x - (float)(dx - 1) * h;
                const unsigned tag = (unsigned)((dz + 1) * 9 + (dy + 1) * 3 + dx) << IDX_BITS;
#pragma unroll 1
                for (int j0 = 0; j0 < nmax; j0 += 32) {
                    const float4 *c = A.recs + (k0[dx] + j0);
                    const int jn = min(32, nmax - j0);
                    unsigned mask = 0;
                    int j = 0;
#pragma unroll 1
                    for (; j < jn; j += U) {
                        float4 r[U];
#pragma unroll
                        for (int i = 0; i < U; ++i) r[i] = c[j + i];
#pragma unroll
                        for (int i = 0; i < U; ++i) {
                            const float v = nl_v(r[i], ox, oy, oz, hi);
                            mask = __funnelshift_l(__float_as_uint(v), mask, 1);
                            near = fminf(near, fabsf(v));
                        }
                    }
                    const int nv = min(32, n[dx] - j0);      // own candidates of this chunk (<= 0: none)
                    mask = nv > 0 ? (mask << (32 - j)) & (0xffffffffu << (32 - nv)) : 0u;
                    while (mask) {
                        const int b = __clz(mask);
                        mask &= ~(0x80000000u >> b);
                        const int t = __float_as_int(c[b].w);
                        const bool take = (t != s) & (t != bp.y) & (t != bp.z);
                        st_pred(out + (size_t)cnt * Mp, (unsigned)t | tag, take & (cnt < maxnb));
                        cnt += take ? 1 : 0;
                    }
                }
            }
        }
    }
    return err | nlist_finish(A, s, m, live, near, cnt, n_out);
}

// Cells [q0, q1) of the stencil of monomer s (melt md, record ri, bonded
// partners bp) in the small resident kernel's buckets: emit(e, take) for every
// candidate, in list order; near: the smallest |v| seen.  Whole warps, at most
// NQ cells, whose counts are in flight together; a cell's first records load
// while the cell before is looked at.
// A bucket's first BUCKET_MAIN records lie in one array, the few further ones
// in another: the walk is bound by the L1 data pipe, which serves one 128-byte
// line at a time, so cells next to each other have to share lines (buckets of
// 512 bytes took 20,000 clocks for 128 monomers of an SM, these take 10,000).
constexpr int BUCKET = 32, BUCKET_MAIN = 4;

template <int NQ, class EMIT>
__device__ __forceinline__ void nlist_cells(const MeltNl &md, int s, bool live, float4 ri, int4 bp, int q0, int q1,
                                            const float4 *brec, const float4 *brec2, const int *count, float &near,
                                            EMIT emit)
{
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int U = BUCKET_MAIN;
    const unsigned code = __float_as_uint(ri.w);
    const int cx = (int)(code & CODE_MASK), cy = (int)((code >> CODE_BITS) & CODE_MASK);
    const int cz = (int)(code >> (2 * CODE_BITS));
    const int nc = md.nc, nbk = md.nbk, cell_off = md.cell_off;
    const float h = md.h, hi = md.hi;
    int cell[NQ], cn[NQ];
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
        const int q = min(q0 + i, 26);
        int zz = cz + q / 9 - 1, yy = cy + (q / 3) % 3 - 1, xx = cx + q % 3 - 1;
        zz = zz < 0 ? nc - 1 : (zz >= nc ? 0 : zz);
        yy = yy < 0 ? nc - 1 : (yy >= nc ? 0 : yy);
        xx = xx < 0 ? nc - 1 : (xx >= nc ? 0 : xx);
        cell[i] = cell_off + ((((zz >> 2) * nbk + (yy >> 2)) * nbk + (xx >> 2)) << 6) +
                  (((zz & 3) << 4) | ((yy & 3) << 2) | (xx & 3));
    }
#pragma unroll
    for (int i = 0; i < NQ; ++i) cn[i] = count[cell[i]];
#pragma unroll
    for (int i = 0; i < NQ; ++i) cn[i] = live && q0 + i < q1 ? cn[i] : 0;
    const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 r[2][U];
#pragma unroll
    for (int k = 0; k < U; ++k) r[0][k] = k < cn[0] ? brec[(size_t)cell[0] * U + k] : none;
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
        const int q = q0 + i, n = cn[i], nmax = __reduce_max_sync(FULL, n);
        if (i + 1 < NQ) {
#pragma unroll
            for (int k = 0; k < U; ++k)
                r[(i + 1) & 1][k] = k < cn[i + 1] ? brec[(size_t)cell[i + 1] * U + k] : none;
        }
        const float ox = ri.x - (float)(q % 3 - 1) * h, oy = ri.y - (float)((q / 3) % 3 - 1) * h,
                    oz = ri.z - (float)(q / 9 - 1) * h;
        auto look = [&](const float4 &c, int j) {
            const float v = nl_v(c, ox, oy, oz, hi);
            const int t = __float_as_int(c.w);
            near = fminf(near, fabsf(v));
            emit((unsigned)t | ((unsigned)q << IDX_BITS),
                 (j < n) & (v < 0.f) & (t != s) & (t != bp.y) & (t != bp.z));
        };
        if (nmax > 0) {
#pragma unroll
            for (int k = 0; k < U; ++k) look(r[i & 1][k], k);
        }
#pragma unroll 1
        for (int j = U; j < nmax; j += 2) {
            const float4 *b = brec2 + (size_t)cell[i] * (BUCKET - U) + (j - U);
            const float4 c0 = j < n ? b[0] : none, c1 = j + 1 < n ? b[1] : none;
            look(c0, j);
            look(c1, j + 1);
        }
    }
}

}  // namespace kg
