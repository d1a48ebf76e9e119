// kg_obs.cu -- observables: <R^2(n)> (the input of the l_K fit, Eq. 14) and
// bond-length / cos(theta) histograms.  Binary64 sums in a fixed order, so
// repeated calls give identical results.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "kg_host.h"

namespace kg {

// <R^2(n)> of short chains in binary64: one thread per chain and lag, one warp
// per block with as many chains as fit (a step of a warp is seven operations of
// the binary64 pipe, 112 clocks of an SM's; four warps a block took 2 us more for
// few chains).  The scaling and the two reductions that the kernel below needs
// first cost about 3 us, which short chains do not earn back.  In us, the former
// binary64 kernel / this / the one below, with the sum over chains: 3 chains of 3
// 8.0 / 8.3 / 10.5, 10 of 20 12.4 / 13.6 / 12.5, 10,000 of 3 692 / 101 / 164, 10,000
// of 20 738 / 197 / 183.
constexpr int R2N_SHORT = 20, R2N_THREADS = 128;

__global__ void __launch_bounds__(32) k_r2n_short(const double *__restrict__ x, long long Mp, int off, int n_ch, int N,
                                                 double *__restrict__ out /* [n_ch][N] */,
                                                 const int *__restrict__ comp_of /* NULL: slot order */)
{
    __shared__ double pos[3][32];
    const int per = 32 / N, c0 = blockIdx.x * per, n_here = min(per, n_ch - c0) * N;
    const int t = threadIdx.x, n = t % N;
    const long long base = (long long)off + (long long)c0 * N;
    if (t < n_here) {
        const long long j = comp_of ? (long long)comp_of[base + t] : base + t;
#pragma unroll
        for (int d = 0; d < 3; ++d) pos[d][t] = x[d * Mp + j];
    }
    __syncwarp();
    if (t >= n_here) return;
    double s = 0.0;
    if (n > 0)
        for (int i = t - n; i + n < t - n + N; ++i) {
            const double dx = pos[0][i + n] - pos[0][i], dy = pos[1][i + n] - pos[1][i], dz = pos[2][i + n] - pos[2][i];
            s += dx * dx + dy * dy + dz * dz;
        }
    out[(size_t)c0 * N + t] = s;
}

// <R^2(n)> of one chain and a share of its lags (block (c, y) of gridDim.y):
// sum_i |x_{i+n} - x_i|^2 for every lag n.  In binary64 the three differences
// and three fused multiply-adds of a pair are 96 clocks of an SM's binary64
// pipe per warp (two lanes a clock), and nothing else counts.  Here a chain's
// positions become 53-bit integers t = (x - x_0) 2^(52-e), 2^e above the chain's
// extent, split as t = 2^30 hi + lo, and a pair's t^2 = 2^60 dhi^2 + 2^31 dhi dlo + dlo^2 is three products a component,
// accumulated as 64-bit integers: dhi^2 exactly, dhi dlo exactly (moved to
// binary64 every R2N_CHUNK terms, before it can overflow), dlo^2 from the upper
// 22 of its 30 bits (2^-21 of a unit of dhi^2).  The quantum, 2^(e-52), is of
// the order of one binary64 ulp at the chain's extent.
// A thread takes W consecutive lags at once: monomer i + n0 + k serves lag
// k of step i and lag k - 1 of step i + 1, so one shared-memory read of a
// position (six words, each array padded by one word in 32 against bank
// conflicts between lanes four monomers apart) serves W pairs.  The window
// at the short end of the lags and its mirror image at the long end go to
// the same thread, so threads have equal work.
// W is 4 where that fills the GPU, where the wide integer multiplies bound it
// (r2n_launch), else 1: four times as many threads with a quarter of the work,
// and a step of one warp alone is a chain of latencies.  In us, binary64 / W = 4 /
// W = 1, with the sum over chains: 20 chains of 100 33 / 45 / 21, 10 of 200 68 /
// 83 / 31, 3 of 1600 2623 / 431 / 149, 100 of 800 712 / 238 / 150; 300 of 800 1351
// / 312 / 350, 1000 of 1600 17802 / 2899 / 3474.  W = 2 is nowhere the best by
// more than 2%.
// A chain with a position that is not finite takes binary64, which says so, and
// so does one whose extent is more than R2N_EXTENT times its shortest bond: the
// quantum goes with the extent and the differences of near monomers are exact in
// binary64 (chains of 1600 at kappa = 3.5 reach about 400; the sums' error stays
// below binary64's for walks, as emulated in 128 bits: 1e-16 against 1e-16 to 5e-16
// for 2 x 20 to 30 x 800; straight rods pass it from 1,500 to 2,000 monomers).
// The row stride Mp is 64-bit: a caller's rows may sit 2^30 or more doubles
// apart, and every index into x is formed in 64-bit arithmetic.
constexpr int R2N_CHUNK = 256;
constexpr float R2N_EXTENT = 2048.0f;

// words of one of the six arrays of a chain of N monomers; sh: padding shift (31: none, the longest chains)
__host__ __device__ __forceinline__ int r2n_words(int N, int sh) { return N + (N >> sh); }

template <int W>
__global__ void __launch_bounds__(R2N_THREADS) k_r2n_chain(const double *__restrict__ x, long long Mp, int off, int N,
                                                          double *__restrict__ out /* [n_ch][N] */,
                                                          const int *__restrict__ comp_of /* NULL: slot order */,
                                                          int sh)
{
    extern __shared__ __align__(16) int words[];   // hi x, y, z, lo x, y, z (first the warps' extents)
    static_assert((R2N_SHORT + 1) * 24 >= 12 * (R2N_THREADS / 32), "the extents and bonds fit the shortest chain's words");
    double *ext_s = reinterpret_cast<double *>(words);
    float *bond_s = reinterpret_cast<float *>(ext_s + R2N_THREADS / 32);
    const int c = blockIdx.x, P = r2n_words(N, sh);
    const long long base = (long long)off + (long long)c * N;
    const long long j0 = comp_of ? (long long)comp_of[base] : base;
    const double o[3] = {x[j0], x[Mp + j0], x[2 * Mp + j0]};
    double ext = 0.0;
    float bond2 = 3.0e38f;                          // the shortest bond, squared
    bool bad = false;
    for (int i = threadIdx.x; i < N; i += R2N_THREADS) {
        const long long j = comp_of ? (long long)comp_of[base + i] : base + i;
        const int i1 = min(i + 1, N - 1);
        const long long j1 = comp_of ? (long long)comp_of[base + i1] : base + i1;
        float b2 = 0.f;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const double xd = x[d * Mp + j], t = fabs(xd - o[d]);
            const float b = f64_to_f32(x[d * Mp + j1] - xd);
            bad |= !isfinite(t);
            ext = fmax(ext, t);
            b2 = fmaf(b, b, b2);
        }
        if (i1 > i) bond2 = fminf(bond2, b2);
    }
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) {
        ext = fmax(ext, __shfl_xor_sync(0xffffffffu, ext, w));
        bond2 = fminf(bond2, __shfl_xor_sync(0xffffffffu, bond2, w));
    }
    if ((threadIdx.x & 31) == 0) {
        ext_s[threadIdx.x >> 5] = ext;
        bond_s[threadIdx.x >> 5] = bond2;
    }
    bad = __syncthreads_or(bad);
#pragma unroll
    for (int w = 0; w < R2N_THREADS / 32; ++w) {
        ext = fmax(ext, ext_s[w]);
        bond2 = fminf(bond2, bond_s[w]);
    }
    __syncthreads();                                // before the words replace them
    bad |= !((float)ext <= R2N_EXTENT * sqrtf(bond2));
    if (blockIdx.y == 0 && threadIdx.x == 0) out[(size_t)c * N] = 0.0;
    if (bad || ext < 1e-200 || ext > 1e200) {       // not finite, a point, or past the scaling's range
        for (int n = 1 + blockIdx.y * R2N_THREADS + threadIdx.x; n < N; n += gridDim.y * R2N_THREADS) {
            double s = 0.0;
            for (int i = 0; i + n < N; ++i) {
                const long long p = comp_of ? (long long)comp_of[base + i] : base + i;
                const long long q = comp_of ? (long long)comp_of[base + i + n] : base + i + n;
                const double dx = x[q] - x[p], dy = x[Mp + q] - x[Mp + p], dz = x[2 * Mp + q] - x[2 * Mp + p];
                s += dx * dx + dy * dy + dz * dz;
            }
            out[(size_t)c * N + n] = s;
        }
        return;
    }
    const int e = ilogb(ext) + 1;
    const double scale = scalbn(1.0, 52 - e);
    for (int i = threadIdx.x; i < N; i += R2N_THREADS) {
        const long long j = comp_of ? (long long)comp_of[base + i] : base + i;
        const int w = i + (i >> sh);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const long long t = __double2ll_rn((x[d * Mp + j] - o[d]) * scale);
            words[d * P + w] = (int)(t >> 30);
            words[(3 + d) * P + w] = (int)(t & ((1 << 30) - 1));
        }
    }
    __syncthreads();
    const double unit = scalbn(1.0, 2 * (e - 52) + 30);
    const int nwin = (N - 1 + W - 1) / W;   // windows of lags 1 + W w ...
    auto get = [&](int i, int *p) {
        const int w = i + (i >> sh);
#pragma unroll
        for (int d = 0; d < 6; ++d) p[d] = words[d * P + w];
    };
    for (int u = blockIdx.y * R2N_THREADS + threadIdx.x; 2 * u < nwin; u += gridDim.y * R2N_THREADS)
        for (int half = 0; half < 2; ++half) {
            const int w = half ? nwin - 1 - u : u;
            if (half && w == u) break;
            const int n0 = 1 + W * w;
            long long hh[W], hl[W], ll[W];
            double mid[W];
            int ring[W][6];                      // monomers i + n0 ... i + n0 + 3, at (i + k) % 4
#pragma unroll
            for (int k = 0; k < W; ++k) {
                hh[k] = hl[k] = ll[k] = 0;
                mid[k] = 0.0;
                if (k) get(min(n0 + k - 1, N - 1), ring[k - 1]);
            }
            auto pair = [&](int k, const int *a, const int *b) {
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const int dh = b[d] - a[d], dl = b[3 + d] - a[3 + d], dq = dl >> 8;
                    hh[k] += (long long)dh * dh;
                    hl[k] += (long long)dh * dl;
                    ll[k] += (long long)dq * dq;
                }
            };
            const int full = max(0, N - n0 - (W - 1));      // steps whose W lags all end in the chain
            int i = 0;
#pragma unroll (W == 1 ? 4 : 1)
            for (; i + W <= full; i += W) {
#pragma unroll
                for (int r = 0; r < W; ++r) {
                    int a[6];
                    get(i + r, a);
                    get(i + r + n0 + W - 1, ring[(r + W - 1) % W]);
#pragma unroll
                    for (int k = 0; k < W; ++k) pair(k, a, ring[(r + k) % W]);
                }
                if ((i & (R2N_CHUNK - 1)) == R2N_CHUNK - W) {
#pragma unroll
                    for (int k = 0; k < W; ++k) {
                        mid[k] += (double)hl[k];
                        hl[k] = 0;
                    }
                }
            }
            for (; i + n0 < N; ++i) {                // the ends, lag by lag (at most 2 W - 2 steps)
                int a[6], p[6];
                get(i, a);
#pragma unroll
                for (int k = 0; k < W; ++k)
                    if (i + n0 + k < N) {
                        get(i + n0 + k, p);
                        pair(k, a, p);
                    }
            }
#pragma unroll
            for (int k = 0; k < W; ++k)
                if (n0 + k < N)
                    out[(size_t)c * N + n0 + k] =
                        ((double)hh[k] * 1073741824.0 + (2.0 * (mid[k] + (double)hl[k]) + (double)ll[k] * 6.103515625e-05)) *
                        unit;                                // 2^30, 2^-14
        }
}

// column sums over chains divided by the number of pairs: R2N_ROWS partial
// sums of every R2N_ROWS-th chain in order, then a fixed tree (500 x 800: 43 ->
// 8 us against one thread per column)
constexpr int R2N_ROWS = 16;

__global__ void __launch_bounds__(32 * R2N_ROWS) k_r2n_reduce(const double *__restrict__ in, int n_ch, int N,
                                                             double *__restrict__ out)
{
    __shared__ double sh[R2N_ROWS][33];
    const int n = blockIdx.x * 32 + threadIdx.x;
    double s = 0.0;
    if (n < N)
        for (int c = threadIdx.y; c < n_ch; c += R2N_ROWS) s += in[(size_t)c * N + n];
    sh[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    for (int w = R2N_ROWS / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.y < w) sh[threadIdx.y][threadIdx.x] += sh[threadIdx.y + w][threadIdx.x];
        __syncthreads();
    }
    if (threadIdx.y == 0 && n < N)
        out[n] = n == 0 ? 0.0 : sh[0][threadIdx.x] / ((double)n_ch * (double)(N - n));
}

// bond-length and cos(theta) counts.  A value's bin is by definition that of
// the binary64 expressions below (min_image_exact and IEEE square roots and
// divides: about 170 binary64 operations a monomer, 180 us for 400,000
// monomers).  The bond vector itself is the plain difference whenever no
// component is near half a box, so three subtractions stay; length and cosine
// in binary32 settle the bin unless they are within their rounding of an
// edge.  Counts go to shared memory first (bins up to HIST_SHARED).  18 us.
constexpr int HIST_SHARED = 4096;
constexpr float HIST_TINY2 = 1e-28f;             // squared lengths from here on keep their digits in binary32

struct Bond64 {
    double v[3];
};

__device__ __noinline__ int hist_bond_exact(Bond64 b, double R0, int nbins)
{
    const double len = sqrt(b.v[0] * b.v[0] + b.v[1] * b.v[1] + b.v[2] * b.v[2]);
    const int k = (int)floor(len / R0 * nbins);
    return k >= 0 && k < nbins ? k : -1;
}

__device__ __noinline__ int hist_cos_exact(Bond64 a, Bond64 b, int nbins)
{
    const double cs = (a.v[0] * b.v[0] + a.v[1] * b.v[1] + a.v[2] * b.v[2])
                      / (sqrt(a.v[0] * a.v[0] + a.v[1] * a.v[1] + a.v[2] * a.v[2])
                         * sqrt(b.v[0] * b.v[0] + b.v[1] * b.v[1] + b.v[2] * b.v[2]));
    const int k = (int)floor((cs + 1.0) * 0.5 * nbins);
    return k < 0 ? 0 : (k >= nbins ? nbins - 1 : k);
}

__global__ void __launch_bounds__(256) k_hist(const double *__restrict__ x, int Mp, int off, int M, int N,
                                             double L, double R0, int nbins, int *__restrict__ bond_h,
                                             int *__restrict__ cos_h, const int *__restrict__ comp_of)
{
    __shared__ int sh[2 * HIST_SHARED];
    const bool local = nbins <= HIST_SHARED;
    int *hb = local ? sh : bond_h, *hc = local ? sh + nbins : cos_h;
    if (local) {
        for (int b = threadIdx.x; b < 2 * nbins; b += blockDim.x) sh[b] = 0;
        __syncthreads();
    }
    const float invL = (float)(1.0 / L), half = (float)(0.49 * L), binsf = (float)nbins, per = (float)((double)nbins / R0);
    // rounding of the binary32 length (relative 3 2^-24, and the bin's) and cosine (absolute 12 2^-24), in bins, doubled
    const float ulp = 5.9604644775390625e-8f, tol = 32.0f * binsf * ulp;
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < M; r += gridDim.x * blockDim.x) {
        const int s = off + r, i = r % N;
        const int j0 = comp_of[s], jm = i >= 1 ? comp_of[s - 1] : j0, jp = i + 1 < N ? comp_of[s + 1] : j0;
        auto bond = [&](int from, int to, Bond64 &b, float3 &f) {
#pragma unroll
            for (int k = 0; k < 3; ++k) b.v[k] = x[(size_t)k * Mp + to] - x[(size_t)k * Mp + from];
            f = make_float3(f64_to_f32(b.v[0]), f64_to_f32(b.v[1]), f64_to_f32(b.v[2]));
            if (!(fmaxf(fmaxf(fabsf(f.x), fabsf(f.y)), fabsf(f.z)) < half)) {
#pragma unroll
                for (int k = 0; k < 3; ++k) b.v[k] = min_image_exact(b.v[k], L, invL);
                f = make_float3(f64_to_f32(b.v[0]), f64_to_f32(b.v[1]), f64_to_f32(b.v[2]));
            }
        };
        if (i + 1 >= N) continue;
        Bond64 b2;
        float3 f2;
        bond(j0, jp, b2, f2);
        const float l2 = fmaf(f2.z, f2.z, fmaf(f2.y, f2.y, f2.x * f2.x));
        {
            const float t = sqrtf(l2) * per;
            int b = t < 2.0f * binsf ? (int)t : nbins;
            const float q = t - (float)b;
            // every value below two histogram widths that sits near an edge, and anything not comparable
            if (!(t >= 2.0f * binsf) && !(q > tol && q < 1.0f - tol)) b = hist_bond_exact(b2, R0, nbins);
            if (b >= 0 && b < nbins) atomicAdd(hb + b, 1);
        }
        if (i >= 1) {
            Bond64 b1;
            float3 f1;
            bond(jm, j0, b1, f1);
            const float l1 = fmaf(f1.z, f1.z, fmaf(f1.y, f1.y, f1.x * f1.x));
            const float cs = fmaf(f1.z, f2.z, fmaf(f1.y, f2.y, f1.x * f2.x)) * rsqrtf(l1) * rsqrtf(l2);
            const float t = (cs + 1.0f) * 0.5f * binsf;
            int b = (int)t;
            const float q = t - (float)b;
            if (!(q > tol && q < 1.0f - tol) || fminf(l1, l2) < HIST_TINY2) b = hist_cos_exact(b1, b2, nbins);
            b = b < 0 ? 0 : (b >= nbins ? nbins - 1 : b);
            atomicAdd(hc + b, 1);
        }
    }
    if (local) {
        __syncthreads();
        for (int b = threadIdx.x; b < nbins; b += blockDim.x) {
            if (sh[b]) atomicAdd(bond_h + b, sh[b]);
            if (sh[nbins + b]) atomicAdd(cos_h + b, sh[nbins + b]);
        }
    }
}

// Dynamic shared memory of k_r2n_chain for chains of N monomers (six words a
// monomer, padded where that fits); above 48 KiB the kernel's opt-in limit is
// raised first.  False if N is too long.
template <int W>
static bool r2n_shared(int N, size_t &smem, int &sh)
{
    sh = 24 * (size_t)r2n_words(N, 5) <= (size_t)R2N_SMEM_MAX ? 5 : 31;
    smem = 24 * (size_t)r2n_words(N, sh);
    if (N < 1 || smem > (size_t)R2N_SMEM_MAX) return false;
    if (smem <= 48 * 1024 - 256) return true;
    return cudaFuncSetAttribute(k_r2n_chain<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess;
}

// blocks of a chain when each thread takes two windows of W lags
template <int W>
static int r2n_split(int N)
{
    const int pairs = ((N - 1 + W - 1) / W + 1) / 2;
    return std::max(1, (pairs + R2N_THREADS - 1) / R2N_THREADS);
}

template <int W>
static bool r2n_chains(const double *x, long long Mp, int off, int n_ch, int N, const int *comp_of, double *tmp,
                       cudaStream_t st)
{
    size_t smem = 0;
    int sh = 5;
    if (!r2n_shared<W>(N, smem, sh)) return false;
    // few chains: the lags of a chain over several blocks, to about eight per SM
    const int split = std::max(1, std::min(r2n_split<W>(N), 152 * 8 / n_ch));
    k_r2n_chain<W><<<dim3(n_ch, split), R2N_THREADS, smem, st>>>(x, Mp, off, N, tmp, comp_of, sh);
    return cudaGetLastError() == cudaSuccess;
}

// <R^2(n)> of n_ch chains of N monomers from x (rows Mp apart); tmp: [n_ch][N]
static bool r2n_launch(const double *x, long long Mp, int off, int n_ch, int N, const int *comp_of, double *tmp,
                       double *out, cudaStream_t st)
{
    if (N <= R2N_SHORT) {
        const int per = 32 / N;
        k_r2n_short<<<(n_ch + per - 1) / per, 32, 0, st>>>(x, Mp, off, n_ch, N, tmp, comp_of);
        if (cudaGetLastError() != cudaSuccess) return false;
    } else {
        // four lags a thread: blocks three quarters full, two or more per SM
        // (300 of 800: 312 against 350 us, 100 of 800: 238 / 150; 1000 of 400,
        // blocks 39% full: 389 / 302)
        const int split = r2n_split<4>(N), pairs = (N + 6) / 8;
        const bool four = 4 * pairs >= 3 * split * R2N_THREADS && (long long)n_ch * split >= 2 * 150;
        if (!(four ? r2n_chains<4>(x, Mp, off, n_ch, N, comp_of, tmp, st)
                   : r2n_chains<1>(x, Mp, off, n_ch, N, comp_of, tmp, st)))
            return false;
    }
    k_r2n_reduce<<<(N + 31) / 32, dim3(32, R2N_ROWS), 0, st>>>(tmp, n_ch, N, out);
    return cudaGetLastError() == cudaSuccess;
}

bool r2n_eval(kg_ctx *c, int melt, double *out_dev)
{
    const MeltDev &md = c->sim.melt[melt];
    c->launches += 2;
    return r2n_launch(c->x, (long long)c->Mp, md.off, md.n_ch, md.N, c->comp_of, c->r2tmp, out_dev, c->stream);
}

void hist_eval(kg_ctx *c, int melt, int nbins, int *out_dev)
{
    const MeltDev &md = c->sim.melt[melt];
    cudaMemsetAsync(out_dev, 0, sizeof(int) * 2 * nbins, c->stream);
    ++c->launches;
    k_hist<<<std::min((md.M + 255) / 256, 152 * 4), 256, 0, c->stream>>>(c->x, c->Mp, md.off, md.M, md.N, md.L, sqrt(c->stage.R0sq),
                                                      nbins, out_dev, out_dev + nbins, c->comp_of);
}

// ---------------------------------------------------------------------------
// ---------------------------------------------------------------------------
// monomer mean-squared displacement (App. B): ref holds, per compute index,
// the position at the last kg_msd_reset plus every box shift a
// double-bridging swap has since added to the unwrapped position, so
// x - ref is the physical displacement
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_msd_reset(const double *__restrict__ x, double *__restrict__ ref, int Mp,
                                                  int off, int M)
{
    const int j = off + blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= off + M) return;
#pragma unroll
    for (int d = 0; d < 3; ++d) ref[(size_t)d * Mp + j] = x[(size_t)d * Mp + j];
}

// block partial sums of |x - ref|^2 in a fixed tree (deterministic)
__global__ void __launch_bounds__(256) k_msd(const double *__restrict__ x, const double *__restrict__ ref, int Mp,
                                            int off, int M, double *__restrict__ part)
{
    __shared__ double sh[256];
    const int j = off + blockIdx.x * blockDim.x + threadIdx.x;
    double s = 0.0;
    if (j < off + M) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const double v = x[(size_t)d * Mp + j] - ref[(size_t)d * Mp + j];
            s += v * v;
        }
    }
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// re-sort of the per-monomer state: ref follows its monomers (out[j] = in[order[j]])
__global__ void __launch_bounds__(256) k_msd_permute(const double *__restrict__ in, double *__restrict__ out,
                                                    const int *__restrict__ order, int Mp, int M)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= M) return;
    const int o = order[j];
#pragma unroll
    for (int d = 0; d < 3; ++d) out[(size_t)d * Mp + j] = in[(size_t)d * Mp + o];
}

static inline int nb256(long long n) { return (int)((n + 255) / 256); }

bool msd_reset(kg_ctx *c, int melt)
{
    if (!c->msd_ref) {
        c->msd_ref = (double *)dev_alloc(c, 6 * (size_t)c->Mp * sizeof(double));
        if (!c->msd_ref) return false;
    }
    const MeltDev &md = c->sim.melt[melt];
    ++c->launches;
    k_msd_reset<<<nb256(md.M), 256, 0, c->stream>>>(c->x, c->msd_ref, c->Mp, md.off, md.M);
    return true;
}

int msd_blocks(const kg_ctx *c, int melt) { return nb256(c->sim.melt[melt].M); }

void msd_eval(kg_ctx *c, int melt, double *part_dev)
{
    const MeltDev &md = c->sim.melt[melt];
    ++c->launches;
    k_msd<<<nb256(md.M), 256, 0, c->stream>>>(c->x, c->msd_ref, c->Mp, md.off, md.M, part_dev);
}

void msd_permute(kg_ctx *c, const int *order)
{
    if (!c->msd_ref) return;
    double *tmp = c->msd_ref + 3 * (size_t)c->Mp;
    c->launches += 1;
    k_msd_permute<<<nb256(c->M), 256, 0, c->stream>>>(c->msd_ref, tmp, order, c->Mp, c->M);
    cudaMemcpyAsync(c->msd_ref, tmp, 3 * (size_t)c->Mp * sizeof(double), cudaMemcpyDeviceToDevice, c->stream);
}

// ---------------------------------------------------------------------------
// static structure factor (App. A): S(q) = |sum_j exp(i q . r_j)|^2 / M for
// q = 2 pi (h, k, l) / L.  The turns of q . r_j are formed exactly: every
// coordinate once as a 64-bit fraction of the box, u = frac(x / L) 2^64, then
// h u_x + k u_y + l u_z in integers modulo 2^64, whose upper word is the
// phase (so unwrapped positions of any size and any (h, k, l) keep their
// precision).  sincospif evaluates it in binary32; the cosines and sines are
// summed as integers of 2^-30 (2^-31 rounding, below the binary32 value's own),
// exactly and in any order.  With the phases, the floor and the sums in
// binary64 the kernel sat on the binary64 pipe (ten of its operations per pair
// of a wave vector and a monomer, two lanes a clock): 256 vectors x 80,000
// monomers took 559 us.
// A thread takes SQ_Q wave vectors, so a monomer's 24 bytes serve that many.
// ---------------------------------------------------------------------------
constexpr int SQ_Q = 4;

__global__ void __launch_bounds__(256) k_sq_turns(const double *__restrict__ x, int Mp, int off, int M, double invL,
                                                 unsigned long long *__restrict__ u, long long *__restrict__ bad)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= M) return;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const double t = x[(size_t)d * Mp + off + r] * invL;
        if (!isfinite(t)) *bad = 1;                        // S is then not a number
        u[(size_t)d * M + r] = __double2ull_rz((t - floor(t)) * 18446744073709551616.0);
    }
}

__global__ void __launch_bounds__(256) k_sq(const unsigned long long *__restrict__ u, int M,
                                           const int *__restrict__ hkl, int nq, long long *__restrict__ part)
{
    const int q0 = blockIdx.x * SQ_Q;
    long long h[SQ_Q], k[SQ_Q], l[SQ_Q], re[SQ_Q], im[SQ_Q];
#pragma unroll
    for (int i = 0; i < SQ_Q; ++i) {
        const int q = min(q0 + i, nq - 1);
        h[i] = hkl[3 * q];
        k[i] = hkl[3 * q + 1];
        l[i] = hkl[3 * q + 2];
        re[i] = im[i] = 0;
    }
    for (int r = blockIdx.y * blockDim.x + threadIdx.x; r < M; r += gridDim.y * blockDim.x) {
        const unsigned long long ux = u[r], uy = u[(size_t)M + r], uz = u[2 * (size_t)M + r];
#pragma unroll
        for (int i = 0; i < SQ_Q; ++i) {
            const unsigned long long t = (unsigned long long)h[i] * ux + (unsigned long long)k[i] * uy +
                                         (unsigned long long)l[i] * uz;
            float sn, cs;
            sincospif((float)(int)(t >> 32) * 4.656612873077392578125e-10f, &sn, &cs);   // half turns: 2^-31
            re[i] += __float2int_rn(cs * 1073741824.0f);
            im[i] += __float2int_rn(sn * 1073741824.0f);
        }
    }
    __shared__ long long sum[2 * SQ_Q];
    if (threadIdx.x < 2 * SQ_Q) sum[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < SQ_Q; ++i) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            re[i] += __shfl_down_sync(0xffffffffu, re[i], o);
            im[i] += __shfl_down_sync(0xffffffffu, im[i], o);
        }
        if ((threadIdx.x & 31) == 0) {
            atomicAdd((unsigned long long *)sum + 2 * i, (unsigned long long)re[i]);
            atomicAdd((unsigned long long *)sum + 2 * i + 1, (unsigned long long)im[i]);
        }
    }
    __syncthreads();
    if (threadIdx.x < 2 * SQ_Q && q0 + (int)threadIdx.x / 2 < nq)
        atomicAdd((unsigned long long *)part + 2 * q0 + threadIdx.x, (unsigned long long)sum[threadIdx.x]);
}

// part[2 nq]: a position was not finite
__global__ void __launch_bounds__(256) k_sq_sum(const long long *__restrict__ part, int nq, int M,
                                               double *__restrict__ S)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nq) return;
    const double re = (double)part[2 * q] * 9.31322574615478515625e-10, im = (double)part[2 * q + 1] * 9.31322574615478515625e-10;
    S[q] = part[2 * nq] ? nan("") : (re * re + im * im) / (double)M;
}

// part_dev: 2 nq + 1 zeroed integers
void sq_eval(kg_ctx *c, int melt, const int *hkl_dev, int nq, long long *part_dev, double *S_dev)
{
    const MeltDev &md = c->sim.melt[melt];
    c->launches += 3;
    unsigned long long *u = (unsigned long long *)c->scratch;
    k_sq_turns<<<nb256(md.M), 256, 0, c->stream>>>(c->x, c->Mp, md.off, md.M, md.invL, u, part_dev + 2 * nq);
    const int nqb = (nq + SQ_Q - 1) / SQ_Q;                // about eight blocks per SM in all
    const int chunks = std::max(1, std::min(nb256(md.M), 152 * 8 / nqb));
    k_sq<<<dim3(nqb, chunks), 256, 0, c->stream>>>(u, md.M, hkl_dev, nq, part_dev);
    k_sq_sum<<<nb256(nq), 256, 0, c->stream>>>(part_dev, nq, md.M, S_dev);
}

// ---------------------------------------------------------------------------
// pair distribution (App. A): pairs with minimum-image distance r < r_max,
// counted in bins of width dr, on the double-bridging cell grid (cells >= 1.3
// sigma, stencil of +-R cells).  A pair's bin is by definition that of the
// binary64 expression ((dx*dx + dy*dy) + dz*dz), dx = d - L rint(d/L), its IEEE
// square root and floor(r / dr).  The binary32 records on that grid (offset
// from the cell corner and cell coordinates) settle it for every pair whose
// r / dr is further than tol from an integer, tol bounding their rounding;
// only the others (~6e-4 of them at dr = 0.01) take the binary64 expression,
// whose divides and square root cost ~100 operations at two lanes a clock:
// with every candidate in binary64 80,000 monomers at r_max = 3 took 11.4 ms.
// Counts are integers, so neither the order nor the two kinds of decision
// show.  Both calls of App. A there (this and 256 wave vectors): 12.1 -> 0.28 ms.
// One thread per monomer in cell order and group of stencil rows: the grid is
// numbered x first, so a row of 2R + 1 cells is one run of records (two where
// it wraps), read in order.  Each pair is counted once, from the half stencil
// (in small boxes, whose rows hold every cell, from the lower position).
// ---------------------------------------------------------------------------
constexpr int GR_MAX_BINS = 2048;

struct GrArgs {
    const float4 *rec;           // records in cell order
    const int *start, *list;     // cell starts; compute index of each position
    const double *x;
    int off, M, Mp, n, cell0, R, nrow, nbins;
    bool all;                    // 2R + 1 >= n: every row holds every cell
    float h, L, invL, inv_dr, tol, cut2;
    double Ld, r_max, dr;
    unsigned long long *hist;
};

__global__ void __launch_bounds__(256) k_gr_sort(const float4 *__restrict__ rec, const int *__restrict__ list, int n,
                                                float4 *__restrict__ out)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n) out[p] = rec[list[p]];
}

// bin of a pair by the binary64 definition (-1: none)
__device__ __noinline__ int gr_exact(const GrArgs &A, int p, int k)
{
    const double r = sqrt(dist2_exact(A.x, A.Mp, A.Ld, A.invL, A.list[p], A.list[k]));
    return r < A.r_max ? (int)__ddiv_rn(r, A.dr) : -1;
}

__global__ void __launch_bounds__(256) k_gr(const __grid_constant__ GrArgs A)
{
    __shared__ unsigned int sh[GR_MAX_BINS];
    for (int b = threadIdx.x; b < A.nbins; b += blockDim.x) sh[b] = 0u;
    __syncthreads();
    const int p = A.off + blockIdx.x * blockDim.x + threadIdx.x;
    if (p < A.off + A.M) {
        const float4 ri = A.rec[p];
        const unsigned code = __float_as_uint(ri.w);
        const int cx = (int)(code & CODE_MASK), cy = (int)((code >> CODE_BITS) & CODE_MASK);
        const int cz = (int)(code >> (2 * CODE_BITS)), n = A.n, R = A.R, w = 2 * R + 1;
        float oy = 0.f, oz = 0.f;
        // records [k0, k1), seen at cell x - cxs from the own one
        auto run = [&](int k0, int k1, int cxs) {
            for (int k = k0; k < k1; ++k) {
                const float4 r = __ldg(A.rec + k);
                const int dc = (int)(__float_as_uint(r.w) & CODE_MASK) - cxs;
                float ex = fmaf((float)dc, A.h, r.x - ri.x), ey = r.y - oy, ez = r.z - oz;
                if (A.all) {
                    ex -= A.L * rintf(ex * A.invL);
                    ey -= A.L * rintf(ey * A.invL);
                    ez -= A.L * rintf(ez * A.invL);
                }
                const float r2 = fmaf(ez, ez, fmaf(ey, ey, ex * ex));
                if (r2 < A.cut2) {
                    const float t = sqrtf(r2) * A.inv_dr;
                    int b = (int)t;
                    const float f = t - (float)b;
                    if (f < A.tol || f > 1.0f - A.tol) b = gr_exact(A, p, k);
                    if ((unsigned)b < (unsigned)A.nbins) atomicAdd(&sh[b], 1u);
                }
            }
        };
        for (int row = blockIdx.y; row < A.nrow; row += gridDim.y) {
            int dy, dz, yy, zz;
            if (A.all) {
                zz = row / n;
                yy = row - zz * n;
                dz = wrap_dk(zz - cz, n);
                dy = wrap_dk(yy - cy, n);
            } else {                                 // dz = 0: dy = 0..R; dz = 1..R: dy = -R..R
                dz = row <= R ? 0 : 1 + (row - R - 1) / w;
                dy = row <= R ? row : (row - R - 1) % w - R;
                zz = cz + dz >= n ? cz + dz - n : cz + dz;
                yy = cy + dy;
                yy = yy < 0 ? yy + n : (yy >= n ? yy - n : yy);
            }
            oy = fmaf((float)-dy, A.h, ri.y);
            oz = fmaf((float)-dz, A.h, ri.z);
            const int *start = A.start + A.cell0 + (zz * n + yy) * n;
            if (A.all) {
                run(max(start[0], p + 1), start[n], cx);
            } else {
                const bool own = row == 0;           // the own row: behind p in its cell, then the cells after it
                const int xa = own ? cx : cx - R, xb = cx + R;
                const int k0 = start[max(xa, 0)], k1 = start[min(xb, n - 1) + 1];
                run(own ? max(k0, p + 1) : k0, k1, cx);
                if (xa < 0) run(start[n + xa], start[n], cx + n);
                if (xb >= n) run(start[0], start[xb - n + 1], cx - n);
            }
        }
    }
    __syncthreads();
    for (int b = threadIdx.x; b < A.nbins; b += blockDim.x)
        if (sh[b]) atomicAdd(A.hist + b, (unsigned long long)sh[b]);
}

// hist_dev: nbins zeroed counts; receives the unordered pairs of each bin
void gr_eval(kg_ctx *c, int melt, int R, double r_max, double dr, int nbins, unsigned long long *hist_dev)
{
    const MeltDev &md = c->sim.melt[melt];
    c->launches += 2;
    k_gr_sort<<<nb256(c->M), 256, 0, c->stream>>>(c->dbrec, c->dblist, c->M, c->recs);   // recs: free between builds
    GrArgs a{};
    a.rec = c->recs;
    a.start = c->dbstart;
    a.list = c->dblist;
    a.x = c->x;
    a.off = md.off;
    a.M = md.M;
    a.Mp = c->Mp;
    a.n = md.ndb;
    a.cell0 = md.dbcell_off;
    a.all = 2 * R + 1 >= md.ndb;
    a.R = R;
    a.nrow = a.all ? md.ndb * md.ndb : (R + 1) + R * (2 * R + 1);
    a.nbins = nbins;
    a.h = md.hdbf;
    a.L = md.Lf;
    a.invL = md.invLf;
    a.Ld = md.L;
    a.r_max = r_max;
    a.dr = dr;
    a.hist = hist_dev;
    // A component adds two offsets (rounded at <= h 2^-24 each), up to Rm + 1
    // cell sides (h itself rounded) and two roundings of a value below (Rm + 2)
    // h, in small boxes an image of L as well; the square root and r / dr add a
    // few roundings of r.  Twice that bound decides.
    const double Rm = a.all ? md.ndb : R, ulp = std::ldexp(1.0, -24);
    const double ec = (3.0 * Rm + 7.0) * md.hdb * ulp + (a.all ? 3.0 * md.L * ulp : 0.0);
    const double er = 2.0 * (std::sqrt(3.0) * ec + 4.0 * r_max * ulp);
    a.inv_dr = (float)(1.0 / dr);
    a.tol = (float)std::min(1.0, er / dr + 4.0 * nbins * ulp);
    a.cut2 = (float)((r_max + er) * (r_max + er) * 1.000001);
    const int nb = nb256(md.M);
    // rows over blocks until about eight blocks per SM are in flight
    const int split = std::max(1, std::min(a.nrow, 152 * 8 / nb));
    k_gr<<<dim3(nb, split), 256, 0, c->stream>>>(a);
}

// <R^2(n)> without any allocation (kg_r2n_noalloc)
// ---------------------------------------------------------------------------
// The per-chain partial sums of k_r2n_chain live in this file-scope array
// instead of a buffer the caller or the library allocates.  Every GPU that
// loads the library holds it (KG_NOALLOC_MAX_MONOMERS doubles, 16 MiB) until
// the process exits.
static __device__ __align__(256) double g_r2n_scratch[KG_NOALLOC_MAX_MONOMERS];

}  // namespace kg

namespace {

// Device address of g_r2n_scratch on the current device.  In host code the
// symbol names a host-side stand-in, not device memory, so it must never be
// handed to a kernel directly.  The address is looked up on every call (the
// lookup allocates nothing), so it stays right after the device's primary
// context has been reset and the module reloaded.
double *scratch_address(kg_status *st)
{
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, kg::g_r2n_scratch) != cudaSuccess) {
        *st = KG_ERR_CUDA;
        return nullptr;
    }
    *st = KG_OK;
    return (double *)p;
}

}  // namespace

extern "C" kg_status kg_r2n_noalloc(const double *x, long long stride, int n_chains, int chain_len, double *out,
                                    void *stream)
{
    if (!x || !out || n_chains < 1 || chain_len < 2 || stride < (long long)n_chains * chain_len)
        return KG_ERR_INVALID_ARG;
    if ((long long)n_chains * chain_len > KG_NOALLOC_MAX_MONOMERS) return KG_ERR_INVALID_ARG;
    if (chain_len > KG_R2N_MAX_CHAIN_LEN) return KG_ERR_INVALID_ARG;
    kg_status st;
    double *scratch = scratch_address(&st);
    if (!scratch) return st;
    return kg::r2n_launch(x, stride, 0, n_chains, chain_len, nullptr, scratch, out, (cudaStream_t)stream) ? KG_OK
                                                                                                         : KG_ERR_CUDA;
}
