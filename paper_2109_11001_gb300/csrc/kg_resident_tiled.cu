// kg_resident_tiled.cu -- the resident MD loop for systems with more monomers
// than threads: one cooperative launch runs K steps, every block walking its
// tiles of 256 monomers in each of them, with the state in memory.
//
// A step is the one-step kernel's tile (kg_step.cuh) and one grid barrier; the
// list rebuild is the counting sort and the list build of the standalone
// kernels between barriers of the same kind.  Every wait is bounded, as in
// kg_resident.cu, and the bits are the same.
//
// It is the default while a block has one tile (194,560 monomers on 152 SMs):
// 100,000 monomers, skin 0.3, n = 2, dt = 0.005: 25.9 -> 17.0 us per step against
// captured graphs of separate launches, whose begin kernel, conditional node
// and gaps cost about 13 us a step.  Beyond that a second round of tiles with
// few of them costs a whole round (199,709 monomers: 39.9 against 34.9 us), and
// the register budget of the hungriest phase (48, five blocks per SM, where the
// one-step kernel has 32 and eight) costs more than the launches (1.6M: 174
// against 148 us); KG_FLAG_PERSISTENT asks for it all the same.
#include <cuda_runtime.h>

#include "kg_resident.cuh"

namespace kg {

constexpr int TILE = 256;

template <int N4>
__global__ void __launch_bounds__(TILE, 5) k_resident_tiled(const __grid_constant__ ResArgs A)
{
    __shared__ float dk[96];
    __shared__ unsigned acc_s[2], out_s;
    __shared__ int wsum[TILE / 16];
    step_block_setup(dk);
    const StepArgs &P = A.st;
    // no block writes the status words before every block has arrived at the last barrier
    const unsigned stop = *(volatile unsigned *)P.flags;
    bool rebuild = *((volatile unsigned *)P.flags + 1) != 0u;
    if (stop) return;                                         // a latched error stops the run
    if (threadIdx.x < 2) acc_s[threadIdx.x] = 0u;
    __syncthreads();
    if ((int)blockIdx.x == A.skip_block) return;              // barrier self-test: never arrives
    GridBar gb{A.bar, acc_s, &out_s, A.spin, 0};
    const long long base = *(volatile long long *)P.stepp;    // the last step run
    const int nthreads = gridDim.x * TILE, first = blockIdx.x * TILE;
    const int nseg = (A.ncell + RES_SEG - 1) / RES_SEG;
    unsigned told = 0, builds = 0;
    for (int it = 0; it < A.K; ++it) {
        const int cur = A.cur0 ^ (it & 1);
        if (rebuild) {                                        // Verlet rebuild; grid-uniform
            for (int s = first + threadIdx.x; s < P.M; s += nthreads) {
                int cell = 0;
                const unsigned err = bin_md_one(*A.sim, s, A.x, A.xb64, A.recb, A.dlt[cur], A.dlt[cur], A.pg[cur], nullptr, nullptr,
                                                A.cellid, A.rank, A.ccount, P.slot_of, &cell);
                if (err) {
                    atomicOr(A.errw, err);
                    gb.note(FAIL);
                } else {                                      // one atomic per segment and warp
                    const int g = cell / RES_SEG;
                    const unsigned act = __activemask(), grp = __match_any_sync(act, g);
                    if ((int)(threadIdx.x & 31) == __ffs(grp) - 1) atomicAdd(A.segtot + g, __popc(grp));
                }
            }
            if ((told = gb.sync()) & (FAIL | GAVE_UP)) break;
            for (int g = blockIdx.x; g < nseg; g += gridDim.x) res_scan_seg<TILE>(A, A.ccount, g, nseg, wsum);
            if ((told = gb.sync()) & GAVE_UP) break;
            for (int s = first + threadIdx.x; s < P.M; s += nthreads) scatter_one(s, A.cellid, A.rank, A.cstart, A.ctmp);
            for (int g = first + threadIdx.x; g < nseg; g += nthreads) A.segtot[g] = 0;   // for the next rebuild
            if ((told = gb.sync()) & GAVE_UP) break;
            for (int p = first + threadIdx.x; p < P.M; p += nthreads)
                if (cellrank_one(p, A.cellid, A.cstart, A.ctmp, A.clist, A.recb, A.recs, A.ccount)) {
                    atomicOr(A.errw, ERR_NL_CAPACITY);
                    gb.note(FAIL);
                }
            if ((told = gb.sync()) & (FAIL | GAVE_UP)) break;
            for (int s0 = first; s0 < P.Mp; s0 += nthreads) {  // whole warps; a row is read by its own thread only
                const unsigned err = nlist_one<false>(A.nl, s0 + threadIdx.x);
                if (err) {
                    atomicOr(A.errw, err);
                    gb.note(FAIL);
                }
            }
            nl_fence();
            ++builds;
        }
        for (int t0 = first; t0 < P.M; t0 += nthreads)
            step_tile<N4, 1, false>(P, t0, A.dlt[cur], A.dlt[cur ^ 1], A.pg[cur], A.pg[cur ^ 1], base + 1 + it, dk,
                                    [&](bool far, unsigned err) {
                                        if (err) atomicOr(A.errw, err);
                                        gb.note((far ? REQ : 0u) | (err ? FAIL : 0u));
                                    },
                                    []() { return true; });
        told = gb.sync();
        rebuild = (told & REQ) != 0u;
        if (told & (FAIL | GAVE_UP)) break;
    }
    if (threadIdx.x == 0 && (told & GAVE_UP)) atomicOr(P.flags, ERR_TIMEOUT);
    if (blockIdx.x == 0 && threadIdx.x == 0) {                // every block has arrived at the last barrier
        if (told & FAIL) atomicOr(P.flags, *(volatile unsigned *)A.errw);
        P.flags[1] = rebuild ? 1u : 0u;
        P.flags[5] += builds;
        if (builds) P.flags[RES_BUILT] = 0u;                  // the cell order is in clist
        *A.stepp = base + A.K;
    }
}

cudaError_t tiled_launch(const ResArgs &a, int n4, int sms, cudaStream_t st)
{
    // a block per tile, or (dilute systems) per segment of the cells that a list
    // build scans, up to what __launch_bounds__ guarantees
    const int nb = std::min(std::max((a.st.M + TILE - 1) / TILE, (a.ncell + RES_SEG - 1) / RES_SEG), 5 * sms);
    return KG_RESIDENT_LAUNCH(k_resident_tiled, n4, nb, TILE, a, st);
}

}  // namespace kg
