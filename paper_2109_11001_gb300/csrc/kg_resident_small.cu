// kg_resident_small.cu -- the resident MD loop (kg_resident.cu) for systems of at
// most 128 monomers per SM, with four threads per monomer.
//
// One warp on a scheduler issues one instruction in four or five clocks (every
// one waits for the one before), so with one thread per monomer a step of a
// small system is a chain of ~2,000 instructions and a list build one of
// ~6,000, on few of the SMs.  Here a block has 64 monomers and four sets of 64
// threads that divide the chain:
//  * a step: set 0 sums the pair terms of list entries 0 .. 7, set 3 forms
//    those of entries 8 .. 15, set 1 the two bond and three angle terms, set 2
//    the noise of the next step; they meet in shared memory, where set 0 adds
//    them in the order of the one-step kernel and updates the monomer;
//  * a list build: each set walks seven of the 27 stencil cells into shared
//    memory, then writes its entries behind those of the sets before it.
// Cells are fixed-size buckets, filled in arrival order and put in order by a
// rank, which saves the scan and the scatter of the counting sort, two phases
// and two grid barriers of a build; a cell with more members than a bucket
// holds sends the build through the counting sort.
//
// Measured per MD step (skin 0.3, n = 12; dt so small that no list is built /
// dt = 0.01, a build every fourth step): 1,000 monomers 3.9 / 7.2 us, 16,000
// 4.5 / 8.6 us, against 4.4 / 11.1 and 4.9 / 12.9 us of one thread per monomer
// (kg_resident.cu) and 25 / 27 us of separate launches.  Blocks of 32 and of
// 128 monomers: 7.1 and 7.6 us at 1,000, 9.3 and 8.6 us at 16,000.  What is
// left of a step without a build are three dependent L2 round trips (gather,
// arrival, poll) and two warps' arithmetic; of a build, the L1 data pipe (the
// walk, 8,000 clocks), binary64 binning (4,000) and two barriers (2,000 each).
//
// (256, 2): at most 128 registers.
#include <cuda_runtime.h>

#include "kg_resident.cuh"

namespace kg {

constexpr int SMALL_SETS = 4;
constexpr int SMALL_THREADS = SMALL_OWN * SMALL_SETS;

// barrier of the threads of set 0
__device__ __forceinline__ void own_sync() { asm volatile("bar.sync 1, %0;" ::"n"(SMALL_OWN) : "memory"); }
constexpr int SMALL_ILP = 8;             // list entries of a set
constexpr int SMALL_EBUF = 16;           // entries a set may find in its cells before the build falls back to one set

struct SmallSmem {
    float dk[96];
    unsigned acc[2], out, overflow;
    int wsum[SMALL_THREADS / 16];
    float near[SMALL_SETS][SMALL_OWN];
    int cnt[SMALL_SETS][SMALL_OWN], total[SMALL_OWN];
    float noise[2][3][SMALL_OWN];                    // by step parity
    union {
        struct {
            float4 pair[SMALL_ILP][SMALL_OWN];       // d and (dU/dr)/r of entries 8 .. 15
            float bond[17][SMALL_OWN];               // (dU/dr)/r and d of two bonds, three angle terms
        } step;
        unsigned ent[SMALL_SETS][SMALL_EBUF][SMALL_OWN];
    };
};

template <int N4>
__global__ void __launch_bounds__(SMALL_THREADS, SMALL_MIN_BLOCKS) k_resident_small(const __grid_constant__ ResArgs A)
{
    __shared__ SmallSmem S;
    step_block_setup(S.dk);
    const StepArgs &P = A.st;
    // no block writes the status words before every block has arrived at the last barrier
    const unsigned stop = *(volatile unsigned *)P.flags;
    bool rebuild = *((volatile unsigned *)P.flags + 1) != 0u;
    int next = (int)*((volatile unsigned *)P.flags + RES_NEXT), built = -1;
    if (stop) return;                                         // a latched error stops the run
    if (threadIdx.x < 2) S.acc[threadIdx.x] = 0u;
    __syncthreads();
    if ((int)blockIdx.x == A.skip_block) return;              // barrier self-test: never arrives
    GridBar gb{A.bar, S.acc, &S.out, A.spin, 0};
    const int set = threadIdx.x / SMALL_OWN, o = threadIdx.x % SMALL_OWN;
    const int s = blockIdx.x * SMALL_OWN + o;
    const bool live = s < P.M;
    const int sv = live ? s : P.M - 1;
    const int nseg = (A.ncell + RES_SEG - 1) / RES_SEG;
    const size_t Mp = (size_t)P.Mp;
    const int Mpi = P.Mp;
    const long long base = *(volatile long long *)P.stepp;    // the last step run
    const int slot = P.slot_of[sv], m = melt_index(P, slot);
    const int4 bp = P.bp[sv];
    const MeltStep &md = P.melt[m];
    const float h = md.h, rc2 = P.rc2;
    const unsigned self = (unsigned)sv | (13u << IDX_BITS);
    const unsigned *col = P.nl + sv;
    int cnt = live ? P.nn[s] : 0;
    float3 v = make_float3(0.f, 0.f, 0.f), d = v;             // set 0
    float4 rb = make_float4(0.f, 0.f, 0.f, 0.f);
    if (live && set == 0) {
        v = make_float3(P.u[s], P.u[Mpi + s], P.u[2 * Mpi + s]);
        const float4 d4 = A.dlt[A.cur0][s];
        d = make_float3(d4.x, d4.y, d4.z);
        rb = A.recb[s];
    }
    unsigned ent[SMALL_ILP];                                  // set 0: entries 0 .. 7, set 3: 8 .. 15
    const int e0 = set == 3 ? SMALL_ILP : 0;
    auto keep = [&]() {
#pragma unroll
        for (int i = 0; i < SMALL_ILP; ++i) ent[i] = e0 + i < cnt ? col[(size_t)(e0 + i) * Mp] : self;
    };
    auto noise = [&](int it) {                                // set 2
        const float3 g = gauss3_f(draw(P.seed, m, 0, (unsigned long long)(base + 1 + it), (uint32_t)(slot - md.off)));
        S.noise[it & 1][0][o] = g.x;
        S.noise[it & 1][1][o] = g.y;
        S.noise[it & 1][2][o] = g.z;
    };
    if (set == 0 || set == 3) keep();
    if (set == 2) noise(0);
    unsigned told = 0, builds = 0;
    for (int it = 0; it < A.K; ++it) {
        const int cur = A.cur0 ^ (it & 1);
        const float4 *pcur = A.pg[cur];
        if (rebuild) {                                        // Verlet rebuild; grid-uniform
            unsigned err = 0;
            int *count = A.count[next], cell = 0, rk = 0;
            if (set == 0 && live) {
                A.dlt[cur][s] = make_float4(d.x, d.y, d.z, 0.f);
                err = bin_md_one(*A.sim, s, A.x, A.xb64, A.recb, A.dlt[cur], A.dlt[cur], A.pg[cur], nullptr, nullptr, A.cellid,
                                 A.rank, count, P.slot_of, &cell, &rk);
                if (err) {
                    atomicOr(A.errw, err);
                    gb.note(FAIL);
                } else if (rk < BUCKET) {
                    A.bidx[(size_t)cell * BUCKET + rk] = s;
                } else {
                    gb.note(OVER);
                }
            }
            if ((told = gb.sync()) & (FAIL | GAVE_UP)) break;
            if (!(told & OVER)) {
                if (set == 0 && live) {
                    const int4 *mem = (const int4 *)(A.bidx + (size_t)cell * BUCKET);
                    const int n = count[cell];
                    int r = 0;
#pragma unroll
                    for (int k = 0; k < BUCKET; k += 4) {     // the count and the first members in flight together
                        if (k >= 12 && k >= n) break;
                        const int4 t = mem[k / 4];
                        r += (k < n && t.x < s) + (k + 1 < n && t.y < s) + (k + 2 < n && t.z < s) + (k + 3 < n && t.w < s);
                    }
                    rb = A.recb[s];
                    float4 *to = r < BUCKET_MAIN ? A.brec + (size_t)cell * BUCKET_MAIN + r
                                                 : A.brec2 + (size_t)cell * (BUCKET - BUCKET_MAIN) + (r - BUCKET_MAIN);
                    *to = make_float4(rb.x, rb.y, rb.z, __int_as_float(s));
                }
                for (int k = blockIdx.x * SMALL_THREADS + threadIdx.x; k < A.ncell; k += gridDim.x * SMALL_THREADS)
                    A.count[next ^ 1][k] = 0;                 // for the next build
                if (threadIdx.x == 0) S.overflow = 0u;
                if ((told = gb.sync()) & GAVE_UP) break;
                const float4 ri = A.recb[sv];
                float near = 3.0e38f;
                int c = 0;
                nlist_cells<7>(A.nl.melt[m], s, live, ri, bp, 7 * set, min(27, 7 * set + 7), A.brec, A.brec2, count,
                               near, [&](unsigned e, bool take) {
                                   if (take && c < SMALL_EBUF) S.ent[set][c][o] = e;
                                   c += take ? 1 : 0;
                               });
                S.cnt[set][o] = c;
                S.near[set][o] = near;
                if (c > SMALL_EBUF) S.overflow = 1u;
                __syncthreads();
                if (S.overflow) {                             // block-uniform: one set walks all 27 cells into the list
                    c = 0;
                    if (set == 0) {
                        auto emit = [&](unsigned e, bool take) {
                            st_pred(A.nl.nl + sv + (size_t)c * Mp, e, take & (c < A.nl.maxnb));
                            c += take ? 1 : 0;
                        };
                        for (int q = 0; q < 27; q += 7)
                            nlist_cells<7>(A.nl.melt[m], s, live, ri, bp, q, min(27, q + 7), A.brec, A.brec2, count,
                                           near, emit);
                    }
                } else {
                    int at = 0;
                    for (int k = 0; k < set; ++k) at += S.cnt[k][o];
                    for (int k = 0; k < c; ++k)
                        if (at + k < A.nl.maxnb) A.nl.nl[s + (size_t)(at + k) * Mp] = S.ent[set][k][o];
                    c = 0;
                    for (int k = 0; k < SMALL_SETS; ++k) {
                        c += S.cnt[k][o];
                        near = fminf(near, S.near[k][o]);
                    }
                    __syncthreads();                          // the rows are whole
                }
                if (set == 0) {
                    err = nlist_finish(A.nl, s, m, live, near, c, cnt);
                    S.total[o] = cnt;
                }
                built = 1 + next;
                next ^= 1;
            } else {                                          // the counting sort of the standalone kernels
                for (int g = blockIdx.x; g < nseg; g += gridDim.x) res_seg_total<SMALL_THREADS>(A, count, g, S.wsum);
                if ((told = gb.sync()) & GAVE_UP) break;
                for (int g = blockIdx.x; g < nseg; g += gridDim.x)
                    res_scan_seg<SMALL_THREADS>(A, count, g, nseg, S.wsum);
                if ((told = gb.sync()) & GAVE_UP) break;
                if (set == 0 && live) scatter_one(s, A.cellid, A.rank, A.cstart, A.ctmp);
                if ((told = gb.sync()) & GAVE_UP) break;
                if (set == 0 && live &&
                    cellrank_one(s, A.cellid, A.cstart, A.ctmp, A.clist, A.recb, A.recs, count)) {   // clears count
                    atomicOr(A.errw, ERR_NL_CAPACITY);
                    gb.note(FAIL);
                }
                if ((told = gb.sync()) & (FAIL | GAVE_UP)) break;
                if (set == 0) {
                    err = nlist_masked<4>(A.nl, s, cnt);
                    S.total[o] = cnt;
                }
                built = 0;
            }
            if (err) {
                atomicOr(A.errw, err);
                gb.note(FAIL);
            }
            __syncthreads();                                  // rows and lengths for every set
            if (set == 3) cnt = S.total[o];
            if (set == 0) {
                d = make_float3(0.f, 0.f, 0.f);
                if (live) rb = A.recb[s];
            }
            if (set == 0 || set == 3) keep();
            ++builds;
        }
        float4 pi = make_float4(rb.x + d.x, rb.y + d.y, rb.z + d.z, rb.w);
        float3 F = make_float3(0.f, 0.f, 0.f);
        const int kmax = __reduce_max_sync(0xffffffffu, cnt);
        if (set == 0 || (set == 3 && kmax > SMALL_ILP)) {
            float4 pj[SMALL_ILP];
#pragma unroll
            for (int i = 0; i < SMALL_ILP; ++i) pj[i] = pcur[ent[i] & IDX_MASK];
            if (set == 3) pi = pcur[sv];
#pragma unroll
            for (int i = 0; i < SMALL_ILP; ++i) {
                const unsigned q = ent[i] >> IDX_BITS;
                const float dx = fmaf(S.dk[q], h, pj[i].x - pi.x);
                const float dy = fmaf(S.dk[32 + q], h, pj[i].y - pi.y);
                const float dz = fmaf(S.dk[64 + q], h, pj[i].z - pi.z);
                const float r2 = fmaf(dz, dz, fmaf(dy, dy, __fmul_rn(dx, dx)));
                float fr = mlj_fr32<N4>(P, r2);
                fr = (e0 + i < cnt && r2 < rc2) ? fr : 0.0f;
                if (set == 0) {
                    F.x = fmaf(fr, dx, F.x); F.y = fmaf(fr, dy, F.y); F.z = fmaf(fr, dz, F.z);
                } else {
                    S.step.pair[i][o] = make_float4(dx, dy, dz, fr);
                }
            }
        } else if (set == 1) {
            unsigned err = 0;
            float t[17];
#pragma unroll
            for (int k = 0; k < 17; ++k) t[k] = 0.f;
            const float4 r0 = bp.x >= 0 ? pcur[bp.x] : pi, r1 = bp.y >= 0 ? pcur[bp.y] : pi;
            const float4 r2 = bp.z >= 0 ? pcur[bp.z] : pi, r3 = bp.w >= 0 ? pcur[bp.w] : pi;
            pi = pcur[sv];
            bonded32<N4>(P, [&](int k, int) { return k == 0 ? r0 : k == 1 ? r1 : k == 2 ? r2 : r3; },
                         [&](int k, float a, float3 x) {
                             if (k < 2) t[k] = a;
                             t[2 + 3 * k] = x.x;
                             t[3 + 3 * k] = x.y;
                             t[4 + 3 * k] = x.z;
                         },
                         md, pi, bp, err);
#pragma unroll
            for (int k = 0; k < 17; ++k) S.step.bond[k][o] = t[k];
            if (err && live) {
                atomicOr(A.errw, err);
                gb.note(FAIL);
            }
        } else if (set == 2 && it + 1 < A.K) {
            noise(it + 1);
        }
        __syncthreads();
        if (set == 0) {
            if (kmax > SMALL_ILP) {
#pragma unroll
                for (int i = 0; i < SMALL_ILP; ++i) {
                    const float4 t = S.step.pair[i][o];
                    F.x = fmaf(t.w, t.x, F.x); F.y = fmaf(t.w, t.y, F.y); F.z = fmaf(t.w, t.z, F.z);
                }
            }
            for (int k = 2 * SMALL_ILP; k < kmax; ++k) {      // few lists are longer
                const unsigned e = k < cnt ? col[(size_t)k * Mp] : self, q = e >> IDX_BITS;
                const float4 p = pcur[e & IDX_MASK];
                const float dx = fmaf(S.dk[q], h, p.x - pi.x);
                const float dy = fmaf(S.dk[32 + q], h, p.y - pi.y);
                const float dz = fmaf(S.dk[64 + q], h, p.z - pi.z);
                const float r2 = fmaf(dz, dz, fmaf(dy, dy, __fmul_rn(dx, dx)));
                float fr = mlj_fr32<N4>(P, r2);
                fr = (k < cnt && r2 < rc2) ? fr : 0.0f;
                F.x = fmaf(fr, dx, F.x); F.y = fmaf(fr, dy, F.y); F.z = fmaf(fr, dz, F.z);
            }
            if (live) {
                auto add = [&](int k, float a) {
                    axpy3(a, make_float3(S.step.bond[2 + 3 * k][o], S.step.bond[3 + 3 * k][o], S.step.bond[4 + 3 * k][o]), F);
                };
                add(0, S.step.bond[0][o]);
                add(1, S.step.bond[1][o]);
                add(2, md.kappa);
                add(3, -md.kappa);
                add(4, md.kappa);
                unsigned err = 0;
                v.x = fmaf(P.dt, fmaf(P.amp, S.noise[it & 1][0][o], fmaf(-P.gamma, v.x, F.x)), v.x);
                v.y = fmaf(P.dt, fmaf(P.amp, S.noise[it & 1][1][o], fmaf(-P.gamma, v.y, F.y)), v.y);
                v.z = fmaf(P.dt, fmaf(P.amp, S.noise[it & 1][2][o], fmaf(-P.gamma, v.z, F.z)), v.z);
                d.x = fmaf(P.dt, v.x, d.x); d.y = fmaf(P.dt, v.y, d.y); d.z = fmaf(P.dt, v.z, d.z);
                A.pg[cur ^ 1][s] = make_float4(rb.x + d.x, rb.y + d.y, rb.z + d.z, rb.w);
                const bool far = fmaf(d.z, d.z, fmaf(d.y, d.y, __fmul_rn(d.x, d.x))) > P.half_skin2;
                if (!isfinite(v.x + v.y + v.z)) err = ERR_NONFINITE;
                if (err) atomicOr(A.errw, err);
                gb.note((far ? REQ : 0u) | (err ? FAIL : 0u));
            }
            own_sync();                                       // the other sets have stored nothing a block could read
            gb.arrive_as_is();
        }
        told = gb.wait();
        rebuild = (told & REQ) != 0u;
        if (told & (FAIL | GAVE_UP)) break;
    }
    const int fin = A.cur0 ^ (A.K & 1);
    if (live && set == 0) {
        A.dlt[fin][s] = make_float4(d.x, d.y, d.z, 0.f);
        P.u[s] = v.x; P.u[Mpi + s] = v.y; P.u[2 * Mpi + s] = v.z;
    }
    if (threadIdx.x == 0 && (told & GAVE_UP)) atomicOr(P.flags, ERR_TIMEOUT);
    if (blockIdx.x == 0 && threadIdx.x == 0) {                // every block has arrived at the last barrier
        if (told & FAIL) atomicOr(P.flags, *(volatile unsigned *)A.errw);
        P.flags[1] = rebuild ? 1u : 0u;
        P.flags[5] += builds;
        if (built >= 0) P.flags[RES_BUILT] = (unsigned)built;
        P.flags[RES_NEXT] = (unsigned)next;
        *A.stepp = base + A.K;
    }
}

cudaError_t small_launch(const ResArgs &a, int n4, cudaStream_t st)
{
    const int nb = (a.st.M + SMALL_OWN - 1) / SMALL_OWN;
    return KG_RESIDENT_LAUNCH(k_resident_small, n4, nb, SMALL_THREADS, a, st);
}

}  // namespace kg
