// kg_step.cu -- the fused MD step of the mixed-precision path (binary32 forces,
// binary64 positions folded from a binary32 displacement at list builds).
//
// One step: U_MLJ^n pair forces over the Verlet list (Eqs. 5-6, truncated and
// shifted at r_c = 2^(1/6)), U_bond^n = U_MLJ^n + FENE bonds (Eq. 10),
// kappa (1 - cos theta) bending (Eq. 4), Langevin friction and Philox noise,
// then the leapfrog update u += dt F, x += dt u (velocity Verlet on the state
// (x_n, u = v_{n-1/2})).
//
// Instruction issue and load latency bound this kernel (its arithmetic per
// byte is low, but the per-entry work of the pair loop is issued for every
// lane of a warp up to the warp's longest list):
//  * every parameter is a by-value kernel argument (constant bank operands,
//    no loads, no registers held for them); a captured graph bakes them in,
//    so graphs are re-captured when the stage changes;
//  * the pair potential is a template on 4n, so each stage of Xi (Eq. 11)
//    gets its own straight-line r^-n;
//  * the pair loop runs to the warp's longest list with per-lane predicates
//    (no divergent loop exits), ILP list entries in flight;
//  * the image shift of an entry's stencil code q is read from three
//    shared-memory word tables of the cell offsets (-1, 0, 1), one per axis
//    (entry q in bank q: conflict-free, three wavefronts where a float4
//    table took about five; the L1 data pipe is this kernel's busiest unit)
//    and scaled by the melt's cell side with one FMA per component;
//  * latency is hidden by resident warps: the pair loop runs before the
//    bonded terms and the noise, holding only its own state, so the kernel
//    fits 32 registers at full occupancy.
#include <cuda_runtime.h>

#include <cmath>

#include "kg_step.cuh"

namespace kg {

// One MD step of every monomer.  (256, 8): at most 32 registers, full
// occupancy (a few bytes spilled after the pair loop).  Measured at 1.6M
// monomers (skin 0.5, n = 12): 94.5 us per launch, against 101.3 at 40
// registers and 97.1 at 48; with the bonded terms before the pair loop it
// needed 48 registers and took 103.5 us.
template <int N4, int TPM>
__global__ void __launch_bounds__(256, 8) k_step32(const __grid_constant__ StepArgs P)
{
    __shared__ float dk[96];
    __shared__ unsigned stop;
    step_block_setup(dk);
    if (threadIdx.x == 0) stop = step_off(P.flags, P.loop, P.k);
    const long long step = *P.stepp + (P.loop ? 1 + P.k : 0);
    step_tile<N4, TPM, true>(P, blockIdx.x * blockDim.x, P.dcur, P.dnext, P.pcur, P.pnext, step, dk,
                             // the rebuild vote per warp (no block barrier: a warp with short
                             // lists leaves without waiting for the block's longest)
                             [&](bool rebuild, unsigned err) {
                                 if (__any_sync(0xffffffffu, rebuild) && (threadIdx.x & 31) == 0) {
                                     if (P.loop) atomicOr(&P.loop->req, 1u << P.k);
                                     else atomicOr(P.flags + 1, 1u);
                                 }
                                 if (err) atomicOr(P.flags, err);
                             },
                             // the block's answer arrives with the first loads of the tile
                             [&]() { __syncthreads(); return !stop; });
}

// 4n of a stage exponent with its own kernel instantiation, 0 otherwise
int n4_of(double n)
{
    const double q = 4.0 * n;
    const int k = (int)std::lround(q);
    if (std::fabs(q - (double)k) > 1e-9) return 0;
    switch (k) {
        case 8: case 12: case 16: case 20: case 23: case 26: case 28:
        case 32: case 36: case 40: case 44: case 48: return k;
        default: return 0;
    }
}

template <int N4>
static void launch_n4(const StepArgs &a, int tpm, int block, long long M, cudaStream_t st)
{
    const int nb = (int)((tpm * M + block - 1) / block);
    if (tpm == 2) k_step32<N4, 2><<<nb, block, 0, st>>>(a);
    else k_step32<N4, 1><<<nb, block, 0, st>>>(a);
}

StepArgs step_args(const kg_ctx *c, int cur)
{
    const StageDev &sg = c->stage;
    StepArgs a{};
    a.recb = c->recb;
    a.dcur = c->dlt[cur];
    a.dnext = c->dlt[cur ^ 1];
    a.pcur = c->pg[cur];
    a.pnext = c->pg[cur ^ 1];
    a.u = (float *)c->u;
    a.nl = c->nl;
    a.nn = c->nn;
    a.slot_of = c->slot_of;
    a.bp = c->bp;
    a.flags = c->flags;
    a.stepp = c->d_step;
    a.seed = c->sim.seed;
    a.M = c->M;
    a.Mp = c->Mp;
    a.n_melts = c->sim.n_melts;
    a.rc2 = c->sim.rc2f;
    a.half_skin2 = c->sim.half_skin2f;
    a.dt = sg.dtf;
    a.gamma = sg.gammaf;
    a.amp = sg.ampf;
    a.c1xn = sg.c1xnf;
    a.c2x6 = sg.c2x6f;
    a.nf = sg.nf;
    a.kf = sg.kfenef;
    a.R0sq = sg.R0sqf;
    a.inv_R0sq = (float)(1.0 / sg.R0sq);
    a.qmin = sg.qminf;
    a.kf_qmin = sg.qmin > 0 ? (float)(sg.kfene / sg.qmin) : 0.0f;
    a.four_R0sq = (float)(4.0 * sg.R0sq);
    for (int m = 0; m < c->sim.n_melts; ++m) {
        const MeltDev &md = c->sim.melt[m];
        a.melt[m] = MeltStep{md.off, md.nc, md.hf, md.Lf, md.invLf, md.kappaf};
    }
    return a;
}

void step_mixed_launch(kg_ctx *c, cudaStream_t st, int cur, LoopDev *loop, int k)
{
    StepArgs a = step_args(c, cur);
    a.loop = loop;
    a.k = k;
    const int tpm = c->tpm, blk = c->block;
    const long long M = c->M;
    switch (n4_of(c->stage.n)) {
        case 8: launch_n4<8>(a, tpm, blk, M, st); break;
        case 12: launch_n4<12>(a, tpm, blk, M, st); break;
        case 16: launch_n4<16>(a, tpm, blk, M, st); break;
        case 20: launch_n4<20>(a, tpm, blk, M, st); break;
        case 23: launch_n4<23>(a, tpm, blk, M, st); break;
        case 26: launch_n4<26>(a, tpm, blk, M, st); break;
        case 28: launch_n4<28>(a, tpm, blk, M, st); break;
        case 32: launch_n4<32>(a, tpm, blk, M, st); break;
        case 36: launch_n4<36>(a, tpm, blk, M, st); break;
        case 40: launch_n4<40>(a, tpm, blk, M, st); break;
        case 44: launch_n4<44>(a, tpm, blk, M, st); break;
        case 48: launch_n4<48>(a, tpm, blk, M, st); break;
        default: launch_n4<0>(a, tpm, blk, M, st); break;
    }
}

}  // namespace kg
