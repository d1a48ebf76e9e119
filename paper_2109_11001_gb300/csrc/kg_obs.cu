// kg_obs.cu -- observables: <R^2(n)> (the input of the l_K fit, Eq. 14) and
// bond-length / cos(theta) histograms.  Binary64 sums in a fixed order, so
// repeated calls give identical results.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "kg_host.h"

namespace kg {

// One block per chain: the chain's unwrapped positions in shared memory;
// thread t accumulates sum_i |x_{i+n} - x_i|^2 for n = t+1, t+1+blockDim, ...
// The row stride Mp is 64-bit: a caller's rows may sit 2^30 or more doubles
// apart, and every index into x is formed in 64-bit arithmetic.
__global__ void __launch_bounds__(256) k_r2n_chain(const double *__restrict__ x, long long Mp, int off, int N,
                                                  double *__restrict__ out /* [n_ch][N] */,
                                                  const int *__restrict__ comp_of /* NULL: slot order */)
{
    extern __shared__ double pos[];          // 3N
    const int c = blockIdx.x;
    const long long base = (long long)off + (long long)c * N;
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const long long j = comp_of ? (long long)comp_of[base + i] : base + i;
        pos[i] = x[j];
        pos[N + i] = x[Mp + j];
        pos[2 * N + i] = x[2 * Mp + j];
    }
    __syncthreads();
    for (int n = threadIdx.x; n < N; n += blockDim.x) {
        double s = 0.0;
        if (n > 0)
            for (int i = 0; i + n < N; ++i) {
                const double dx = pos[i + n] - pos[i], dy = pos[N + i + n] - pos[N + i],
                             dz = pos[2 * N + i + n] - pos[2 * N + i];
                s += dx * dx + dy * dy + dz * dz;
            }
        out[(size_t)c * N + n] = s;
    }
}

// column sums over chains, in chain order, divided by the number of pairs
__global__ void __launch_bounds__(256) k_r2n_reduce(const double *__restrict__ in, int n_ch, int N,
                                                   double *__restrict__ out)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    double s = 0.0;
    for (int c = 0; c < n_ch; ++c) s += in[(size_t)c * N + n];
    out[n] = n == 0 ? 0.0 : s / ((double)n_ch * (double)(N - n));
}

__global__ void __launch_bounds__(256) k_hist(const double *__restrict__ x, int Mp, int off, int M, int N,
                                             double L, double R0, int nbins, int *__restrict__ bond_h,
                                             int *__restrict__ cos_h, const int *__restrict__ comp_of)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= M) return;
    const int s = off + r, i = r % N;
    const int j0 = comp_of[s], jm = i >= 1 ? comp_of[s - 1] : j0, jp = i + 1 < N ? comp_of[s + 1] : j0;
    double b1[3], b2[3];
    if (i + 1 < N) {
#pragma unroll
        for (int k = 0; k < 3; ++k) b2[k] = min_image_exact(x[k * Mp + jp] - x[k * Mp + j0], L);
        const double len = sqrt(b2[0] * b2[0] + b2[1] * b2[1] + b2[2] * b2[2]);
        const int b = (int)floor(len / R0 * nbins);
        if (b >= 0 && b < nbins) atomicAdd(bond_h + b, 1);
    }
    if (i >= 1 && i + 1 < N) {
#pragma unroll
        for (int k = 0; k < 3; ++k) b1[k] = min_image_exact(x[k * Mp + j0] - x[k * Mp + jm], L);
        const double cs = (b1[0] * b2[0] + b1[1] * b2[1] + b1[2] * b2[2])
                          / (sqrt(b1[0] * b1[0] + b1[1] * b1[1] + b1[2] * b1[2])
                             * sqrt(b2[0] * b2[0] + b2[1] * b2[1] + b2[2] * b2[2]));
        int b = (int)floor((cs + 1.0) * 0.5 * nbins);
        b = b < 0 ? 0 : (b >= nbins ? nbins - 1 : b);
        atomicAdd(cos_h + b, 1);
    }
}

// Dynamic shared memory of k_r2n_chain for chains of N monomers (3N doubles);
// above 48 KiB the kernel's opt-in limit is raised first.
bool r2n_smem_ready(int N)
{
    const size_t smem = sizeof(double) * 3 * (size_t)N;
    if (N < 1 || smem > (size_t)R2N_SMEM_MAX) return false;
    if (smem <= 48 * 1024) return true;
    return cudaFuncSetAttribute(k_r2n_chain, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess;
}

bool r2n_eval(kg_ctx *c, int melt, double *out_dev)
{
    const MeltDev &md = c->sim.melt[melt];
    if (!r2n_smem_ready(md.N)) return false;
    c->launches += 2;
    k_r2n_chain<<<md.n_ch, 256, sizeof(double) * 3 * md.N, c->stream>>>(c->x, (long long)c->Mp, md.off, md.N,
                                                                          c->r2tmp, c->comp_of);
    if (cudaGetLastError() != cudaSuccess) return false;
    k_r2n_reduce<<<(md.N + 255) / 256, 256, 0, c->stream>>>(c->r2tmp, md.n_ch, md.N, out_dev);
    return cudaGetLastError() == cudaSuccess;
}

void hist_eval(kg_ctx *c, int melt, int nbins, int *out_dev)
{
    const MeltDev &md = c->sim.melt[melt];
    cudaMemsetAsync(out_dev, 0, sizeof(int) * 2 * nbins, c->stream);
    ++c->launches;
    k_hist<<<(md.M + 255) / 256, 256, 0, c->stream>>>(c->x, c->Mp, md.off, md.M, md.N, md.L, sqrt(c->stage.R0sq),
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
    const double r = sqrt(dist2_exact(A.x, A.Mp, A.Ld, A.list[p], A.list[k]));
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
    const cudaStream_t s = (cudaStream_t)stream;
    const size_t smem = sizeof(double) * 3 * chain_len;
    if (!kg::r2n_smem_ready(chain_len)) return KG_ERR_CUDA;
    kg::k_r2n_chain<<<n_chains, 256, smem, s>>>(x, stride, 0, chain_len, scratch, nullptr);
    kg::k_r2n_reduce<<<(chain_len + 255) / 256, 256, 0, s>>>(scratch, n_chains, chain_len, out);
    return cudaGetLastError() == cudaSuccess ? KG_OK : KG_ERR_CUDA;
}

