// kg_internal.cuh -- device-side data layout and helpers of the GB300 DBH library.
//
// Layout in HBM (all melts of a context are concatenated slot ranges):
//   x        double[3][Mp]   canonical unwrapped positions (SoA)
//   u        float[3][Mp] (mixed) / double[3][Mp] (FP64): state velocity v_{n-1/2}
//   pid      int[Mp]         particle ids carried through double-bridging swaps
//   recb     float4[Mp]      build-time position record: offset from the corner
//                            of its Verlet-grid cell + packed cell coordinates
//   dlt[2]   float4[Mp]      (mixed) displacement since the last build, ping-pong
//   pg[2]    float4[Mp]      gather record of the step: recb + displacement, code
//                            (binary64: for the near-pair test)
//   pos64[2] double4_32a[Mp] (FP64) gather copy of the positions, ping-pong
//   xb       double4_32a[Mp] (FP64) positions at the last build
//   nl       uint[maxnb][Mp] Verlet list, column-major (coalesced per k); an
//                            entry is j | q << IDX_BITS, q the stencil cell
//                            (image shift) of j relative to the owner's cell
//   nn       int[Mp]         list lengths
// Mp is the total slot count rounded up to a multiple of 32.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace kg {

constexpr int MAX_MELTS = 64;
constexpr int CODE_BITS = 10;           // cells per axis on the code grid <= 1024
constexpr int CODE_MASK = (1 << CODE_BITS) - 1;
constexpr int MAX_CELL_OCC = 1024;      // a cell holding more monomers is reported, never scanned
constexpr int IDX_BITS = 27;            // Verlet-list entry: index bits, then the 5-bit stencil code
constexpr unsigned IDX_MASK = (1u << IDX_BITS) - 1u;
constexpr int SHIFT_SLOTS = 32;         // shift-table entries per melt (27 used)

// device error / status word bits
enum : unsigned {
    ERR_OVERSTRETCH = 1u,
    ERR_NONFINITE = 2u,
    ERR_NL_CAPACITY = 4u,
    ERR_DB_CAPACITY = 8u,
    ERR_TIMEOUT = 16u,
    ERR_DB_INTERNAL = 32u,
};

constexpr int LOOP_MAX = 16;             // steps in the body of a captured step loop, at most (multiple of 4)

// State of a captured step loop (kg_md.cu) on the device.
struct LoopDev {
    long long rem;           // steps still to run
    int n;                   // of them in the present pass of the loop body
    int src;                 // buffer that holds the state when the pass begins (1 only before a list build)
    int par;                 // buffer that holds it after the last pass
    unsigned req;            // bit k: step k of the pass asked for a list rebuild (later ones of the pass are skipped)
};

// Non-zero if step k of a pass (or a step launched by itself, lp null) does not
// run: a latched error, the end of the loop, or a build asked for by an earlier
// step of the pass (this step's own bit may already be set by another block).
// The three words are loaded together.
__device__ __forceinline__ unsigned step_off(const unsigned *flags, const LoopDev *lp, int k)
{
    const unsigned err = *(const volatile unsigned *)flags;
    if (!lp) return err;
    const volatile LoopDev *v = lp;
    const int n = v->n;
    const unsigned req = v->req;
    return err | (unsigned)(k >= n) | (req & ((1u << k) - 1u));
}

// Ends a pass of `len` steps: counts the steps done (those up to the first
// that asked for a build), passes the request on (flags[1]) and returns true if
// another pass has to run.  flags[6] counts the pass's kernels other than these
// steps: six of the build chain, the end kernel, steps that returned at once.
__device__ __forceinline__ bool loop_finish(LoopDev *lp, int len, long long *stepp, unsigned *flags)
{
    const int done = lp->req ? min(lp->n, __ffs((int)lp->req)) : lp->n;
    stepp[0] += done;
    const long long rem = lp->rem - done;
    const bool more = rem > 0 && !flags[0];
    lp->rem = rem;
    lp->n = (int)(rem < len ? rem : len);
    lp->src = done & 1;                        // every pass starts in buffer 0, or with a build that writes it
    lp->par = more ? 0 : done & 1;
    flags[1] = lp->req ? 1u : 0u;
    lp->req = 0u;
    flags[6] += 7 + len - done;
    return more;
}

// status words kept by the resident MD kernel: how the last Verlet build left the
// cell order (0: clist; 1 + b: buckets with counts b), and the zeroed count buffer
constexpr int RES_BUILT = 8, RES_NEXT = 9;

struct MeltDev {
    int off, M, N, n_ch;          // slots [off, off+M): chain c, position i -> off + c*N + i
    int ch_off;                   // chains of earlier melts (global chain index = ch_off + c)
    double L, invL, kappa;
    float Lf, invLf, kappaf;
    // Verlet-list cell grid (cells >= r_c + skin), numbered brick-major
    // (4x4x4-cell bricks) so that a block of consecutive monomers in cell
    // order has a compact neighbourhood; the position records are offsets
    // from the corners of these cells
    int nc, nbk, cell_off;
    double h, invh;
    float hf;
    float nl_lo, nl_hi;      // binary32 prefilter: r^2 < nl_lo in, r^2 >= nl_hi out
    float near2;             // binary64 step: pairs with r^2 >= near2 on the gather records lie beyond r_c
    // double-bridging grid (cells >= db_bond_max); binary32 records on it decide
    // the swap-bond criterion outside the band [db_lo, db_hi) around db_bond_max^2
    int ndb, dbcell_off;
    double hdb, invhdb;
    float hdbf, db_lo, db_hi;
};

// Parameters of the current potential stage (Eqs. 6, 9, 10) and thermostat.
struct StageDev {
    double n, c1, c2;        // U_MLJ^n(r) = c1 r^-n - c2 r^-6 + 1  (r < r_c)
    double kfene, R0sq;      // FENE: -k R0^2/2 ln(1 - r^2/R0^2)
    double qmin, r2star, ustar;  // continuation beyond r*^2 = (1 - qmin) R0^2 (qmin > 0)
    double dt, gamma, T, amp;  // amp = sqrt(2 gamma T / dt)
    float nf, c1f, c2f, kfenef, R0sqf, dtf, gammaf, ampf, qminf, r2starf, ustarf;
    float c2x6f, c1xnf;      // 6 c2 and n c1: fr = (6 c2 r^-6 - n c1 r^-n) / r^2
    int nkind;               // 0: general n, 1: integer n, 2: n = 5.75, 3: n = 6.5
    int nint;
};

struct SimDev {
    MeltDev melt[MAX_MELTS];
    int n_melts, M, Mp, maxnb;
    double rc2, rl2, db_lim2;
    float rc2f, half_skin2f;
    unsigned long long seed;
    int paper_metropolis;
};

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): 10 rounds of two
// 32x32->64 multiplies with multipliers 0xD2511F53, 0xCD9E8D57 and a Weyl key
// schedule with increments 0x9E3779B9, 0xBB67AE85.
// Counter layout: (index, time_lo, time_hi, melt<<4 | purpose), key = seed.
// Purposes: 0 MD noise (index = melt-local slot, time = step),
//           1 DB attempt draw, 2 DB partner draw (index = attempt, time = sweep).
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
        k.x += 0x9E3779B9u;
        k.y += 0xBB67AE85u;
    }
    return c;
}

__device__ __forceinline__ uint4 draw(unsigned long long seed, int melt, unsigned purpose,
                                      unsigned long long time, uint32_t index)
{
    return philox4x32_10(make_uint4(index, (uint32_t)time, (uint32_t)(time >> 32),
                                    ((uint32_t)melt << 4) | purpose),
                         make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
}

// (2*(w>>9)+1) * 2^-24: a uniform in (0,1), exact in binary32 and binary64.
__device__ __forceinline__ float unit_open_f(uint32_t w)
{
    return __uint2float_rn(2u * (w >> 9) + 1u) * 5.9604644775390625e-8f;
}
__device__ __forceinline__ double unit_open_d(uint32_t w)
{
    return (double)(2u * (w >> 9) + 1u) * 5.9604644775390625e-8;
}

// Three standard normals by Box-Muller.
__device__ __forceinline__ float3 gauss3_f(uint4 r)
{
    const float a = sqrtf(-2.0f * logf(unit_open_f(r.x)));
    const float b = sqrtf(-2.0f * logf(unit_open_f(r.z)));
    float s, c;
    sincospif(2.0f * unit_open_f(r.y), &s, &c);
    return make_float3(a * c, a * s, b * cospif(2.0f * unit_open_f(r.w)));
}
__device__ __forceinline__ double3 gauss3_d(uint4 r)
{
    const double a = sqrt(-2.0 * log(unit_open_d(r.x)));
    const double b = sqrt(-2.0 * log(unit_open_d(r.z)));
    double s, c;
    sincospi(2.0 * unit_open_d(r.y), &s, &c);
    return make_double3(a * c, a * s, b * cospi(2.0 * unit_open_d(r.w)));
}

// floor(w * n / 2^64): exact integer map of a 64-bit word onto [0, n).
__device__ __forceinline__ long long mul_hi64(unsigned long long w, unsigned long long n)
{
    return (long long)__umul64hi(w, n);
}

// ---------------------------------------------------------------------------
// geometry
// ---------------------------------------------------------------------------
__device__ __forceinline__ int melt_of(const SimDev &S, int s)
{
    int m = 0;
    while (m + 1 < S.n_melts && s >= S.melt[m + 1].off) ++m;
    return m;
}

__device__ __forceinline__ unsigned pack_code(int cx, int cy, int cz)
{
    return (unsigned)cx | ((unsigned)cy << CODE_BITS) | ((unsigned)cz << (2 * CODE_BITS));
}

__device__ __forceinline__ int wrap_dk(int dk, int n)
{
    if (dk > n / 2) dk -= n;
    else if (dk < -(n / 2)) dk += n;
    return dk;
}

// Verlet-grid cell index of cell coordinates (cx, cy, cz), brick-major.
__device__ __forceinline__ int md_cell(const MeltDev &md, int cx, int cy, int cz)
{
    return md.cell_off + ((((cz >> 2) * md.nbk + (cy >> 2)) * md.nbk + (cx >> 2)) << 6) +
           (((cz & 3) << 4) | ((cy & 3) << 2) | (cx & 3));
}

// Conversions between binary64, binary32 and integers in 32-bit integer
// instructions, for the ordinary range of their arguments; the rest takes the
// conversion instruction.  A binary64 conversion or rounding occupies the
// binary64 pipe, two lanes a clock per SM here, like an addition: 16 clocks a
// warp, where these take 5 to 15 instructions of the 128-lane integer and
// logic pipes.  Same results as the instructions, bit for bit.
__device__ __forceinline__ double f32_to_f64(float f)
{
    const unsigned u = __float_as_uint(f), a = u & 0x7fffffffu;
    if (a - 0x00800000u >= 0x7f000000u) return (double)f;            // zero, subnormal, infinite or NaN
    return __hiloint2double((int)((u & 0x80000000u) | ((a >> 3) + (896u << 20))), (int)(u << 29));
}

__device__ __forceinline__ float f64_to_f32(double d)                // to nearest even
{
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const unsigned e = (hi >> 20) & 0x7ffu;
    if (e - 897u >= 253u) return __double2float_rn(d);               // outside [2^-126, 2^127) in size
    const unsigned long long r = (((unsigned long long)hi << 32) | lo) + 0x0fffffffu + ((lo >> 29) & 1u);
    return __uint_as_float((__funnelshift_l((unsigned)r, (unsigned)(r >> 32), 3) - (0x180u << 23)) | (hi & 0x80000000u));
}

// floor(p) as an integer; g: the same as binary64
__device__ __forceinline__ int floor_f64(double p, double &g)
{
    const unsigned hi = (unsigned)__double2hiint(p), lo = (unsigned)__double2loint(p);
    const int e = (int)((hi >> 20) & 0x7ffu) - 1023;
    if ((unsigned)e >= 30u) {                                        // below 1 or from 2^30 in size, infinite, NaN
        if (e < 0) {
            g = (hi >> 31) && ((hi << 1) | lo) ? -1.0 : 0.0;
            return (int)g;
        }
        g = floor(p);
        return (int)g;
    }
    const unsigned m = __funnelshift_l(lo, hi, 11) | 0x80000000u;    // the significand's top 32 bits: [1, 2) 2^31
    unsigned t = m >> (31 - e);
    if (hi >> 31) t += ((m << (e + 1)) | (lo << 11)) != 0u;          // away from zero below it
    const int z = __clz((int)t);                                     // t in [1, 2^30]
    const unsigned n = t << z;
    g = __hiloint2double((int)((hi & 0x80000000u) | ((unsigned)(1023 + 31 - z) << 20) | ((n << 1) >> 12)), (int)(n << 21));
    return hi >> 31 ? -(int)t : (int)t;
}

// Cell of a binary64 coordinate on a grid of n cells of side h = L / n per
// period: g = floor(x / h) of the unwrapped coordinate, taken modulo n, and
// the offset x - g h from that cell's corner, rounded once to binary32.
// n h differs from L by at most an ulp of L, so the offsets of monomers in
// different periodic images stay consistent to ~1e-14 sigma.  Two binary64
// operations, each explicitly rounded so that every kernel inlining it
// computes the same bits; floor and conversions in integer instructions.
__device__ __forceinline__ int cell_of(double x, double h, double invh, int n, float &off)
{
    double g;
    const int k = floor_f64(__dmul_rn(x, invh), g);
    off = f64_to_f32(__fma_rn(-g, h, x));
    const int c = k % n;
    return c < 0 ? c + n : c;
}

// Number of box lengths that a minimum image takes off d, rint(d / L), in
// binary32 where that settles it: the binary32 quotient is good to 2e-3 below
// 1e4 box lengths, so 0.02 from a half its nearest integer is the binary64
// one's.  `sure` false: it does not (or d is not finite).
__device__ __forceinline__ float image_of(double d, float invL, bool &sure)
{
    const float y = f64_to_f32(d) * invL, k = rintf(y);
    sure = fabsf(y - k) < 0.48f && fabsf(y) < 1e4f;
    return k;
}

// d - L*rint(d/L) as written, no contraction.  Most vectors here join
// monomers of the same image (k = 0 leaves d as it is) or near ones, so the
// binary64 divide and rounding, ~12 of the thin pipe's operations, are rarely
// taken.
__device__ __forceinline__ double min_image_exact(double d, double L, float invL)
{
    bool sure;
    const float k = image_of(d, invL, sure);
    if (!sure) return __dsub_rn(d, __dmul_rn(L, rint(__ddiv_rn(d, L))));
    return k == 0.f ? d : __dsub_rn(d, __dmul_rn(L, f32_to_f64(k)));
}

// squared binary64 distance between slots s and t, ((dx*dx + dy*dy) + dz*dz)
__device__ __forceinline__ double dist2_exact(const double *__restrict__ x, int Mp, double L, float invL, int s, int t)
{
    const double dx = min_image_exact(__dsub_rn(x[t], x[s]), L, invL);
    const double dy = min_image_exact(__dsub_rn(x[Mp + t], x[Mp + s]), L, invL);
    const double dz = min_image_exact(__dsub_rn(x[2 * Mp + t], x[2 * Mp + s]), L, invL);
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// Minimum-image vector from gather record i to gather record j (binary32):
// p = offset from the build-time cell corner + displacement, w = packed cell
// coordinates.  The cell difference, wrapped to the nearest image, carries
// the integer part, so no large-magnitude value enters the sum.  The wrap is
// unambiguous while |true cell difference| < nc/2, which holds when nc >= 11
// for every pair closer than 6 sigma (two bonds at the 2 R0 error limit,
// cells >= 1.37 sigma, up to half a skin of drift each); smaller grids (small
// boxes) finish with an explicit minimum image of the small vector.
__device__ __forceinline__ float3 rec_rel(float4 pi, float4 pj, int nc, float h, float L, float invL)
{
    const unsigned ci = __float_as_uint(pi.w), cj = __float_as_uint(pj.w);
    const int dkx = wrap_dk((int)(cj & CODE_MASK) - (int)(ci & CODE_MASK), nc);
    const int dky = wrap_dk((int)((cj >> CODE_BITS) & CODE_MASK) - (int)((ci >> CODE_BITS) & CODE_MASK), nc);
    const int dkz = wrap_dk((int)(cj >> (2 * CODE_BITS)) - (int)(ci >> (2 * CODE_BITS)), nc);
    float3 d = make_float3((pj.x - pi.x) + (float)dkx * h, (pj.y - pi.y) + (float)dky * h,
                           (pj.z - pi.z) + (float)dkz * h);
    if (nc < 11) {
        d.x -= L * rintf(d.x * invL);
        d.y -= L * rintf(d.y * invL);
        d.z -= L * rintf(d.z * invL);
    }
    return d;
}

}  // namespace kg
