// kg_db.cuh -- device pieces shared by the uniform and the learned
// double-bridging sweeps: candidate enumeration in a topology view, the
// bond / bending terms of a swap, and the ordered commit.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>

#include "kg_gridbar.cuh"
#include "kg_host.h"

namespace kg {

constexpr int CAND_CAP = 48;

struct Cand {
    int key, key2, kind, d, q;
};

struct DBC {
    const double *__restrict__ x;
    int Mp;
    const int *__restrict__ pid;
    const int *__restrict__ cell;
    const int *__restrict__ start;
    const int *__restrict__ list;
    const float4 *__restrict__ rec;    // binary32 records on the 1.3 sigma grid (k_bin_db)
    MeltDev md;
    int melt;
    double lim2, kfene, R0, T, qmin, nexp;
};

// topology view: slot -> monomer (occ) and monomer -> slot (cur)
struct ViewMap {
    const int *o;
    const int *c;
    __device__ __forceinline__ int occ(int s) const { return o[s]; }
    __device__ __forceinline__ int cur(int p) const { return c[p]; }
};

// Slot relabelling of one swap; the same map takes x -> x' and x' -> x.
__device__ __forceinline__ int swap_slot(int s, int kind, int A, int B, int pA, int pB, int N, int off)
{
    const int r = s - off, ch = r / N, i = r - ch * N;
    if (kind == 0) {
        if (i > pA) {
            if (ch == A) return off + B * N + i;
            if (ch == B) return off + A * N + i;
        }
    } else {
        if (ch == A && i > pA) return off + B * N + (N - 1 - i);
        if (ch == B && i <= pB) return off + A * N + (N - 1 - i);
    }
    return s;
}

template <class V>
struct ViewMove {
    V b;
    int kind, A, B, pA, pB, N, off;
    __device__ __forceinline__ int occ(int s) const { return b.occ(swap_slot(s, kind, A, B, pA, pB, N, off)); }
    __device__ __forceinline__ int cur(int p) const { return swap_slot(b.cur(p), kind, A, B, pA, pB, N, off); }
};

__device__ __forceinline__ double d2(const DBC &C, int a, int b) { return dist2_exact(C.x, C.Mp, C.md.L, C.md.invLf, a, b); }

// Swap-bond criterion d2(a, b) <= 1.3^2, decided exactly: the binary32 record
// distance settles every pair outside the band [db_lo, db_hi), which bounds
// its rounding error; pairs inside it take the binary64 distance.
__device__ __forceinline__ bool within(const DBC &C, int a, int b)
{
    const float3 d = rec_rel(__ldg(C.rec + a), __ldg(C.rec + b), C.md.ndb, C.md.hdbf, C.md.Lf, C.md.invLf);
    const float r2 = d.x * d.x + d.y * d.y + d.z * d.z;
    if (r2 < C.md.db_lo) return true;
    if (r2 >= C.md.db_hi) return false;
    return d2(C, a, b) <= C.lim2;
}

// the acceptance uniform of attempt k
__device__ __forceinline__ double accept_u(unsigned long long seed, int melt, long long sweep, int k)
{
    const uint4 r = draw(seed, melt, 1, (unsigned long long)sweep, (uint32_t)k);
    return ((double)(r.z >> 5) * 67108864.0 + (double)(r.w >> 6)) * (1.0 / 9007199254740992.0);
}

// per-warp candidate scratch of one partner enumeration
struct __align__(16) WarpCand {
    Cand tmp[CAND_CAP];
    Cand cand[CAND_CAP];
    int n;
};

constexpr unsigned FULL_MASK = 0xffffffffu;

// Admissible partners P(b) of bond (c, b) in view v, one warp: lane q < 27
// scans stencil cell q around the bond's lower monomer.  With ORDER the list
// is left in wc.cand ordered by (key, key2) (the monomer ids of the monomer
// that would bond to the drawn bond's lower end and of the partner bond's
// other monomer).  Returns |P|, or -1 (error bit set) on a capacity overflow.
template <bool ORDER, class V>
__device__ int warp_partners(const DBC &C, const V &v, int c, int b, WarpCand &wc, unsigned &err)
{
    const int lane = threadIdx.x & 31;
    const MeltDev &md = C.md;
    const int N = md.N;
    const int us = md.off + c * N + b;
    const int pu = v.occ(us), pw = v.occ(us + 1);
    if (!within(C, pu, pw)) return 0;
    if (lane == 0) wc.n = 0;
    __syncwarp();
    bool bad = false;
    if (lane < 27) {
        // the record names the cell; list entries, and then their slots, are
        // loaded four at a time: an evaluation is a chain of L2 round trips
        const int n = md.ndb;
        const unsigned code = __float_as_uint(__ldg(C.rec + pu).w);
        const int cx = (int)(code & CODE_MASK), cy = (int)((code >> CODE_BITS) & CODE_MASK);
        const int cz = (int)(code >> (2 * CODE_BITS));
        const int dz = lane / 9 - 1, dy = (lane / 3) % 3 - 1, dx = lane % 3 - 1;
        const int cell = md.dbcell_off + (((cz + dz + n) % n) * n + (cy + dy + n) % n) * n + (cx + dx + n) % n;
        const int b0 = C.start[cell], e = C.start[cell + 1];
        if (e - b0 > MAX_CELL_OCC) {
            bad = true;
        } else {
            int tt[4], sl[4];
            for (int k = b0; k < e; ++k) {
                if (((k - b0) & 3) == 0) {
#pragma unroll
                    for (int u = 0; u < 4; ++u) tt[u] = C.list[min(k + u, e - 1)];
#pragma unroll
                    for (int u = 0; u < 4; ++u) sl[u] = v.cur(tt[u]);
                }
                const int u = (k - b0) & 3;
                const int t = u == 0 ? tt[0] : u == 1 ? tt[1] : u == 2 ? tt[2] : tt[3];
                const int ts = u == 0 ? sl[0] : u == 1 ? sl[1] : u == 2 ? sl[2] : sl[3];
                const int r = ts - md.off, d = r / N, i = r - d * N;
                if (d == c) continue;
                if (i != b + 1 && i != N - 2 - b) continue;   // neither kind can use t
                if (!within(C, pu, t)) continue;
                if (i == b + 1) {                          // kind 0: t = D_{b+1}
                    const int up = v.occ(md.off + d * N + b);
                    if (within(C, up, pw) && within(C, up, t)) {
                        const int pos = atomicAdd(&wc.n, 1);
                        if (ORDER && pos < CAND_CAP) wc.tmp[pos] = Cand{C.pid[t], C.pid[up], 0, d, b};
                    }
                }
                if (i == N - 2 - b) {                      // kind 1: t = D_q, q = N-2-b
                    const int t1 = v.occ(ts + 1);
                    if (within(C, t1, pw) && within(C, t, t1)) {
                        const int pos = atomicAdd(&wc.n, 1);
                        if (ORDER && pos < CAND_CAP) wc.tmp[pos] = Cand{C.pid[t], C.pid[t1], 1, d, i};
                    }
                }
            }
        }
    }
    __syncwarp();
    const int n = wc.n;
    if (__any_sync(FULL_MASK, bad) || n > CAND_CAP) {
        err |= ERR_DB_CAPACITY;
        return -1;
    }
    if (ORDER) {
        for (int j = lane; j < n; j += 32) {       // rank by the (unique) key pair
            const Cand cj = wc.tmp[j];
            int r = 0;
            for (int i = 0; i < n; ++i) {
                const Cand ci = wc.tmp[i];
                r += (ci.key < cj.key) || (ci.key == cj.key && ci.key2 < cj.key2);
            }
            wc.cand[r] = cj;
        }
        __syncwarp();
    }
    return n;
}

// FENE log term of a bond of length r (kg_params.fene_qmin continuation beyond r*)
__device__ __forceinline__ double fene_of_r(const DBC &C, double r)
{
    const double q = 1.0 - (r / C.R0) * (r / C.R0);
    if (C.qmin > 0.0 && q < C.qmin)           // continuation beyond r* (kg_params.fene_qmin)
        return -0.5 * C.kfene * C.R0 * C.R0 * log(C.qmin) + C.kfene * (r * r - (1.0 - C.qmin) * C.R0 * C.R0) / (2.0 * C.qmin);
    return -0.5 * C.kfene * C.R0 * C.R0 * log(q);
}

template <class V>
__device__ double bond_fene(const DBC &C, const V &v, int chain, int idx)
{
    const int s = C.md.off + chain * C.md.N + idx;
    return fene_of_r(C, sqrt(d2(C, v.occ(s), v.occ(s + 1))));
}

// cos of the angle at vertex i of `chain` in view v (1 at a chain end)
template <class V>
__device__ double vcos(const DBC &C, const V &v, int chain, int i)
{
    const int N = C.md.N;
    if (i < 1 || i > N - 2) return 1.0;
    const int s = C.md.off + chain * N + i;
    const int a = v.occ(s - 1), b = v.occ(s), c = v.occ(s + 1);
    const double L = C.md.L;
    double b1[3], b2[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        b1[k] = min_image_exact(C.x[k * C.Mp + b] - C.x[k * C.Mp + a], L, C.md.invLf);
        b2[k] = min_image_exact(C.x[k * C.Mp + c] - C.x[k * C.Mp + b], L, C.md.invLf);
    }
    return (b1[0] * b2[0] + b1[1] * b2[1] + b1[2] * b2[2])
           / (sqrt(b1[0] * b1[0] + b1[1] * b1[1] + b1[2] * b1[2])
              * sqrt(b2[0] * b2[0] + b2[1] * b2[1] + b2[2] * b2[2]));
}

template <class V>
__device__ double bend(const DBC &C, const V &v, int chain, int i)
{
    if (i < 1 || i > C.md.N - 2) return 0.0;
    return C.md.kappa * (1.0 - vcos(C, v, chain, i));
}

// v or the topology after a swap, chosen per lane
template <class V>
struct ViewEither {
    ViewMove<V> m;
    bool moved;
    __device__ __forceinline__ int occ(int s) const
    {
        return m.b.occ(moved ? swap_slot(s, m.kind, m.A, m.B, m.pA, m.pB, m.N, m.off) : s);
    }
};

__device__ __forceinline__ DBC make_dbc(const SimDev &S, const StageDev &st, int m, const double *x,
                                        const int *pid, const int *cell, const int *start, const int *list,
                                        const float4 *rec, double T)
{
    DBC C;
    C.x = x; C.Mp = S.Mp; C.pid = pid; C.cell = cell; C.start = start; C.list = list; C.rec = rec;
    C.md = S.melt[m]; C.melt = m; C.lim2 = S.db_lim2; C.kfene = st.kfene; C.R0 = sqrt(st.R0sq); C.T = T; C.qmin = st.qmin;
    C.nexp = st.n;
    return C;
}

// ---------------------------------------------------------------------------
// Ordered commit in rounds.  Every attempt record carries the number of swaps
// committed (in its melt) when it was evaluated; chains and cells of the 1.3
// sigma grid carry the number of the last commit that touched them (chain_ver,
// cell_ver; -1 for none).  A record is stale when a commit at or after its
// version touched one of its two chains, or stamped a cell within P::radius
// cells of one of its junction monomers: only then can its evaluation differ,
// since swaps preserve positions, the bonds inside moved segments and the
// lengths of the pieces on either side of every bond.
// One round: (A) every stale record at or after the melt's position is
// re-evaluated against the current topology, across the whole GPU; (B) the
// first accepted attempt of each melt from its position (every record there is
// now current) is committed: one block rewrites the slot maps and adds the
// box shifts, all blocks stamp cells; or, if there is none, the melt is
// finished (statistics).  Rounds repeat until every melt is finished: as many
// rounds as accepted swaps plus one, and the result is that of the strictly
// sequential loop over attempts.
// All rounds run in one cooperative launch, two grid barriers a round, the
// second of which also says whether a melt is left.  An evaluation is a long
// chain of dependent loads and binary64 operations, and a round waits for its
// slowest one, so it is cut in two: the draw and the partner scan of the drawn
// bond, one warp per record (most sets are empty, and done); then, for a
// non-empty set, E::TASKS independent parts on as many warps.  160,000
// attempts of a 1.6M-monomer melt: about 30 us a round (14 swaps 526 us, 21 swaps
// 668, 25 swaps 790), against about 60 as two launches a round with the host
// reading the finished flags now and then, an attempt evaluated by one warp and
// the dE of a swap by one lane.
// round[RS m + 0..5] of one of two buffers (by round parity: commits write the
// next round's while every block reads this one's) = position, commits,
// finished, re-evaluations, the first accepted attempt at or after the position
// (INT_MAX: none), empty records.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool stale_rec(int4 head, int4 cells, const int *chain_ver, int choff, const int *cell_ver)
{
    const int v = head.w;
    int newest = chain_ver[choff + head.y];                    // loads of one latency, then one comparison
    if (head.x & 1) newest = max(newest, chain_ver[choff + head.z]);
    if (cells.x >= 0) newest = max(newest, cell_ver[cells.x]);
    if (cells.y >= 0) newest = max(newest, cell_ver[cells.y]);
    if (cells.z >= 0) newest = max(newest, cell_ver[cells.z]);
    if (cells.w >= 0) newest = max(newest, cell_ver[cells.w]);
    return newest >= v;
}

struct RoundArgs {
    const SimDev *sim;
    const double *x;
    const int *cell, *koff;
    Attempt *att;
    int *occ, *curmap, *img, *chain_ver, *cell_ver;
    int *round;                  // [2][MAX_MELTS][RS]
    int *old;                    // [2 M]: slot maps of the two chains of a commit, per melt
    long long *stats;
    unsigned *flags;
    unsigned *errw;              // error bits of this launch (zero at launch), the evaluator's among them
    unsigned long long *bar;     // three barrier words, zero at launch
    unsigned spin;
    long long most;              // rounds (attempts + 1)
};

// (A) by blocks of THREADS records.  E provides, each for one whole warp,
//   scan(m, k, g, Attempt &a): draw attempt k (global index g) of melt m and its partner; flags 0, or 1 | 4
//   task(m, a, t): part t < TASKS of deciding a, as a binary64 value
// and for one thread accepts(m, k, a, const double *parts).
template <int THREADS, class E>
__device__ void restale_pass(E &ev, const RoundArgs &R, int *round, bool first)
{
    __shared__ int todo[THREADS], und[THREADS], n_todo, n_und;
    __shared__ double part[THREADS][E::TASKS];
    const SimDev &S = *R.sim;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int NW = THREADS / 32;
    const int Ktot = R.koff[S.n_melts];
    auto melt = [&](int k) {
        int m = 0;
        while (k >= R.koff[m + 1]) ++m;
        return m;
    };
    for (int base = blockIdx.x * THREADS; base < Ktot; base += gridDim.x * THREADS) {
        const int k = base + threadIdx.x;
        bool st = false, un = false, acc = false, empty = false;
        int m = 0;
        if (threadIdx.x == 0) n_todo = n_und = 0;
        if (k < Ktot) {
            m = melt(k);
            const int *rd = round + RS * m;
            if (!rd[2] && k - R.koff[m] >= rd[0]) {
                const int4 *rec = reinterpret_cast<const int4 *>(R.att + k);
                const int4 head = rec[0], cells = rec[1];
                st = stale_rec(head, cells, R.chain_ver, S.melt[m].ch_off, R.cell_ver);
                un = !st && (head.x & 4);
                acc = !st && (head.x & 2);
                empty = !(head.x & 1);
            }
        }
        // fresh records are current: note the first accepted one of each melt (and, once, count the empty ones)
        const int m0 = __shfl_sync(FULL_MASK, m, 0);
        if (__all_sync(FULL_MASK, k >= Ktot || m == m0)) {       // one melt in the warp: one atomic
            const int f = __reduce_min_sync(FULL_MASK, acc ? k - R.koff[m] : INT_MAX);
            const int ne = __popc(__ballot_sync(FULL_MASK, empty));
            if (lane == 0 && f != INT_MAX) atomicMin(round + RS * m0 + 4, f);
            if (lane == 0 && first && ne) atomicAdd(round + RS * m0 + 5, ne);
        } else {
            if (acc) atomicMin(round + RS * m + 4, k - R.koff[m]);
            if (first && empty) atomicAdd(round + RS * m + 5, 1);
        }
        if (!__syncthreads_or(st || un)) continue;
        if (st) todo[atomicAdd(&n_todo, 1)] = k;
        if (un) und[atomicAdd(&n_und, 1)] = k;
        __syncthreads();
        for (int i = warp; i < n_todo; i += NW) {
            const int kk = todo[i], mm = melt(kk);
            Attempt a;
            ev.scan(mm, kk - R.koff[mm], kk, a);
            if (lane == 0) {
                const int was = R.att[kk].flags & 1, is = a.flags & 1;
                a.ver = round[RS * mm + 1];
                R.att[kk] = a;
                atomicAdd(round + RS * mm + 3, 1);
                if (was != is) atomicAdd(round + RS * mm + 5, was - is);
                if (is) und[atomicAdd(&n_und, 1)] = kk;
            }
            __syncwarp();
        }
        __syncthreads();
        const int nu = n_und;
        for (int i = warp; i < nu * E::TASKS; i += NW) {
            const int kk = und[i / E::TASKS], t = i % E::TASKS;
            const double v = ev.task(melt(kk), R.att[kk], t);
            if (lane == 0) part[i / E::TASKS][t] = v;
            __syncwarp();
        }
        __syncthreads();
        if ((int)threadIdx.x < nu) {
            const int kk = und[threadIdx.x], mm = melt(kk);
            const bool yes = ev.accepts(mm, kk - R.koff[mm], R.att[kk], part[threadIdx.x]);
            R.att[kk].flags = yes ? 3 : 1;
            if (yes) atomicMin(round + RS * mm + 4, kk - R.koff[mm]);
        }
        __syncthreads();
    }
}

// (B) every block; block m % gridDim.x rewrites melt m's maps.  P provides
// radius.  nx: the next round's state.  True while the melt is unfinished.
template <class P>
__device__ bool commit_pass(P &pol, const RoundArgs &A, int m, const int *round, int *next)
{
    __shared__ int sh[6];
    const SimDev &S = *A.sim;
    const int tid = threadIdx.x;
    const int *R = round + RS * m;
    int *X = next + RS * m;
    const MeltDev &md = S.melt[m];
    const int N = md.N, off = md.off, Mp = S.Mp;
    const int k0 = A.koff[m], K = A.koff[m + 1] - k0;
    const bool mine = m % (int)gridDim.x == (int)blockIdx.x;
    const int found = min(R[4], K);                // the first accepted attempt at or after the position
    const int nc = R[1];
    if (R[2] || found == K) {                      // the melt is finished
        if (mine && tid == 0) {
            if (!R[2]) {
                A.stats[4 * m + 0] = K;
                A.stats[4 * m + 1] = R[5];
                A.stats[4 * m + 2] = nc;
                A.stats[4 * m + 3] = R[3];
                if (nc) atomicOr(A.flags + 1, 1u);
            }
            X[2] = 1;
        }
        return false;
    }
    const Attempt &a = A.att[k0 + found];
    const int Rr = pol.radius(md);
    // stamp the cells within Rr of the four junction monomers, over the grid
    const int n = md.ndb, W = 2 * Rr + 1;
    for (int t = blockIdx.x * blockDim.x + tid; t < 4 * W * W * W; t += gridDim.x * blockDim.x) {
        const int q = t / (W * W * W), r = t - q * W * W * W;
        const int cq = a.cell[q];
        if (cq < 0) continue;
        const int c0 = cq - md.dbcell_off;
        const int cx = c0 % n, cy = (c0 / n) % n, cz = c0 / (n * n);
        const int dx = r % W - Rr, dy = (r / W) % W - Rr, dz = r / (W * W) - Rr;
        const int xx = ((cx + dx) % n + n) % n, yy = ((cy + dy) % n + n) % n;
        const int zz = ((cz + dz) % n + n) % n;
        A.cell_ver[md.dbcell_off + (zz * n + yy) * n + xx] = nc;
    }
    if (!mine) return true;
    const int kind = a.kind, cA = a.A, cB = a.B, pA = a.pA, pB = a.pB;
    const int baseA = off + cA * N, baseB = off + cB * N;
    // box shifts of the moved segments; segment 0: A' slots pA+1..N-1 anchored at A' slot pA; segment 1: kind 0 ->
    // B' slots pA+1..N-1 at pA, kind 1 -> B' slots 0..pB at pB+1 (maps still before the swap)
    if (tid < 6) {
        const int seg = tid / 3, d = tid % 3;
        const int fs = seg == 0 ? baseA + pA + 1 : (kind == 0 ? baseB + pA + 1 : baseB + pB);
        const int as = seg == 0 ? baseA + pA : (kind == 0 ? baseB + pA : baseB + pB + 1);
        const int f = A.occ[swap_slot(fs, kind, cA, cB, pA, pB, N, off)];
        const int an = A.occ[swap_slot(as, kind, cA, cB, pA, pB, N, off)];
        sh[tid] = -((int)rint(__ddiv_rn(__dsub_rn(A.x[d * Mp + f], A.x[d * Mp + an]), md.L))
                    + A.img[d * Mp + f] - A.img[d * Mp + an]);
    }
    // new slot maps: read whole before they are written, PER entries of a
    // thread in registers (all loads in flight together); longer chains go
    // through a copy of the two chains' maps
    constexpr int PER = 16;
    const bool copy = 2 * N > PER * (int)blockDim.x;
    int *old_occ = A.old + 2 * off;
    int val[PER];
    if (copy) {
        for (int j = tid; j < 2 * N; j += blockDim.x) old_occ[j] = A.occ[j < N ? baseA + j : baseB + (j - N)];
    } else {
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int j = tid + q * blockDim.x;
            if (j < 2 * N)
                val[q] = A.occ[swap_slot(j < N ? baseA + j : baseB + (j - N), kind, cA, cB, pA, pB, N, off)];
        }
    }
    __syncthreads();
    auto moved = [&](int j, int p) {                 // entry j of the two chains is now monomer p
        const int s = j < N ? baseA + j : baseB + (j - N);
        A.occ[s] = p;
        A.curmap[p] = s;
        const int jj = j - N;
        const int seg = j < N ? (j > pA ? 0 : -1) : (((kind == 0 && jj > pA) || (kind == 1 && jj <= pB)) ? 1 : -1);
        if (seg >= 0) {
#pragma unroll
            for (int d = 0; d < 3; ++d)
                if (sh[3 * seg + d]) A.img[d * Mp + p] += sh[3 * seg + d];
        }
    };
    if (copy) {
        for (int j = tid; j < 2 * N; j += blockDim.x) {
            const int src = swap_slot(j < N ? baseA + j : baseB + (j - N), kind, cA, cB, pA, pB, N, off);
            moved(j, src - baseA < N && src >= baseA ? old_occ[src - baseA] : old_occ[N + src - baseB]);
        }
    } else {
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int j = tid + q * blockDim.x;
            if (j < 2 * N) moved(j, val[q]);
        }
    }
    if (tid == 0) {
        A.chain_ver[md.ch_off + cA] = nc;
        A.chain_ver[md.ch_off + cB] = nc;
        X[0] = found + 1;
        X[1] = nc + 1;
        X[2] = 0;
        X[3] = R[3];
        X[4] = INT_MAX;                            // to be found again by the next pass (A)
        X[5] = R[5];
    }
    __syncthreads();                               // sh is used again for the next melt
    return true;
}

// All rounds of a sweep; every block of a cooperative launch (ev, pol as above).
// Errors of the evaluations go to a word of this launch, so the status word is
// the same for a block however late it starts: block 0 writes it after a
// barrier at which every block has arrived.  A round that saw an error ends the
// sweep before its commit.
template <int THREADS, class E, class P>
__device__ void rounds_body(E &ev, P &pol, const RoundArgs &R)
{
    __shared__ unsigned acc_s[2], out_s, stop_s;
    if (threadIdx.x < 2) acc_s[threadIdx.x] = 0u;
    if (threadIdx.x == 0) stop_s = *(volatile unsigned *)R.flags;
    __syncthreads();
    if (stop_s) return;                                        // a latched error stops the sweep
    GridBar gb{R.bar, acc_s, &out_s, R.spin, 0};
    unsigned told = 0;
    for (long long r = 0; r <= R.most; ++r) {
        int *round = R.round + (r & 1) * RS * MAX_MELTS, *next = R.round + ((r + 1) & 1) * RS * MAX_MELTS;
        restale_pass<THREADS>(ev, R, round, r == 0);
        if (threadIdx.x == 0 && *(volatile unsigned *)R.errw) gb.note(FAIL);
        if ((told = gb.sync()) & (FAIL | GAVE_UP)) break;
        bool left = false;
        for (int m = 0; m < R.sim->n_melts; ++m) left |= commit_pass(pol, R, m, round, next);
        if (threadIdx.x == 0 && left) gb.note(REQ);
        told = gb.sync();
        if (!(told & REQ) || (told & GAVE_UP)) break;
    }
    if (threadIdx.x == 0 && (told & GAVE_UP)) atomicOr(R.flags, ERR_TIMEOUT);
    if (blockIdx.x == 0 && threadIdx.x == 0 && (told & FAIL)) atomicOr(R.flags, *(volatile unsigned *)R.errw);
}

RoundArgs round_args(kg_ctx *c);                // kg_db.cu

constexpr unsigned ROUNDS_SPIN = 1u << 24;         // barrier polls (0.32 us apart) before giving up

// Launches kernel K (blocks of `threads`, smem bytes, RoundArgs in r, then the
// evaluator's arguments) on as many blocks as the attempts need and the GPU holds.
template <class KERNEL, class... ARGS>
cudaError_t rounds_launch(kg_ctx *c, KERNEL K, int threads, size_t smem, long long tot, int nm, RoundArgs r, ARGS... args)
{
    int dev = 0, nsm = 0, per = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, K, threads, smem);
    if (e != cudaSuccess) return e;
    if (per < 1) return cudaErrorCooperativeLaunchTooLarge;
    const long long want = (tot + threads - 1) / threads;      // a thread looks at one record
    const long long nb = std::min((long long)per * nsm, std::max((long long)nm, std::max(want, 1LL)));
    e = cudaMemsetAsync(c->dbbar, 0, 4 * sizeof(unsigned long long), c->stream);   // and the error word
    if (e != cudaSuccess) return e;
    r.bar = c->dbbar;
    r.spin = ROUNDS_SPIN;
    r.most = tot;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)nb);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = c->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    c->launches += 1;
    return cudaLaunchKernelEx(&cfg, K, r, args...);
}

}  // namespace kg
