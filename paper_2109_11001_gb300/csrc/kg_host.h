// kg_host.h -- host-side context of the GB300 DBH library (internal).
#pragma once
#include <cuda_runtime.h>

#include <functional>
#include <vector>

#include "kg.h"
#include "kg_internal.cuh"

struct kg_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    kg_allocator alloc{};
    bool have_alloc = false;

    kg_params p{};
    std::vector<kg_melt> melts;
    int precision = KG_FP64;
    int M = 0, Mp = 0;           // slots, padded slots

    kg::SimDev sim{};            // host copy
    kg::SimDev *d_sim = nullptr;
    kg::StageDev stage{};        // host copy of the stage in force
    kg::StageDev *d_stage = nullptr;

    std::vector<kg_stage> schedule;
    size_t stage_idx = 0;
    long long stage_left = -1;   // < 0: open-ended
    long long step = 0, sweep = 0;
    double t_since_sweep = 0.0;
    std::vector<double> carry;   // fractional DB attempts per melt
    kg_status latched = KG_ERR_STATE;

    // state
    double *x = nullptr;         // [3][Mp]; mixed: current only outside kg_step (see xb64)
    double *xb64 = nullptr;      // mixed: binary64 positions at the last Verlet build [3][Mp];
                                 // the current position is xb64 + dlt[cur] (folded at every
                                 // build and at the end of every kg_step call)
    void *u = nullptr;           // [3][Mp] float or double
    int *pid = nullptr;          // particle id of the monomer at each compute index
    int *slot_of = nullptr;      // compute index -> chain-major slot
    int *comp_of = nullptr;      // chain-major slot -> compute index
    int4 *bp = nullptr;          // compute indices of slots s-2, s-1, s+1, s+2 (-1 past a chain end)
    bool clist_valid = false;    // the last Verlet build's cell order can seed a re-sort
    bool sort_after_load = false;  // re-sort after the first build that follows a load
    long long since_sort = 0;
    long long *d_step = nullptr;   // device step counter (index of the step being run)
    bool d_step_stale = true;      // host must write it before the next step
    cudaStream_t cap_stream = nullptr;
    cudaEvent_t order_ev = nullptr;    // follow_default
    cudaGraphExec_t gexec[kg::LOOP_MAX / 4] = {};   // captured step loops with bodies of 4, 8, 12 and 16 steps
    bool graph_failed = false;
    kg::LoopDev *loop = nullptr;   // their state on the device
    double build_every = 8.0;      // MD steps between Verlet builds in the last call long enough to tell
    unsigned builds_seen = 0;      // builds counted on the device up to the end of the last call
    unsigned long long *resbar = nullptr;   // barrier words, error word and segment totals of the resident launch
    int *bcount = nullptr, *bidx = nullptr; // its cell buckets: two sets of counts, members in arrival order
    float4 *brec = nullptr;                 // and records in order
    bool buckets = false;
    int res_sms = -1;            // SMs of the GPU (< 0: not asked yet)
    bool resident_failed = false;
    long long sort_interval = 200;
    int block = 128;             // threads per block of the fused step kernel
    int tpm = 1;                 // threads per monomer of the mixed step kernel (1 or 2)
    float4 *recb = nullptr;      // build records: offset from the Verlet-cell corner, cell coordinates
    float4 *recs = nullptr;      // the same in cell order (Verlet-list build)
    float4 *dlt[2] = {nullptr, nullptr};   // (mixed) displacement since the build
    float4 *pg[2] = {nullptr, nullptr};    // gather records recb + displacement (binary64: for the near-pair test)
    float4 *shtab = nullptr;     // image shift of each stencil code, SHIFT_SLOTS per melt
    double4_32a *pos64[2] = {nullptr, nullptr};
    double4_32a *xb = nullptr;
    int cur = 0;                 // ping-pong index of the gather buffer in use

    // Verlet list and its cell grid
    int ncell_md = 0;
    int *cellid = nullptr, *rank = nullptr, *ccount = nullptr, *cstart = nullptr, *clist = nullptr;
    int *ctmp = nullptr;         // cell-ordered list before the in-cell ranking
    int *bsum = nullptr;         // scan block sums (shared by both grids)
    int maxnb = 0;
    unsigned *nl = nullptr;      // entries j | stencil code << IDX_BITS
    int *nn = nullptr;

    // double-bridging
    int ncell_db = 0;
    int *dbcell = nullptr, *dbrank = nullptr, *dbcount = nullptr, *dbstart = nullptr, *dblist = nullptr;
    float4 *dbrec = nullptr;     // binary32 records on the DB grid (swap-bond prefilter)
    int *dbmark = nullptr;       // per DB cell: number of the last commit of the sweep near it (-1: none)
    int *chain_ver = nullptr;    // per chain: number of the last commit of the sweep that touched it
    int n_chain_total = 0;
    int *dbround = nullptr;      // per melt: position, commits, finished, re-evaluations
    void *att = nullptr;         // kg::Attempt[att_cap]
    long long att_cap = 0;
    int *koff = nullptr;         // [n_melts+1] attempt offsets
    unsigned long long *dbbar = nullptr;   // grid-barrier words of the commit rounds, and their error word
    int *img = nullptr;
    long long *db_stats = nullptr;   // [n_melts][4]

    // learned proposal (kg_mlp.cu, kg_learned.cu)
    float *mlp_master = nullptr;         // binary32 master weights [KG_MLP_NPARAM]
    float *mlp_adam = nullptr;           // Adam moments m, v [2][KG_MLP_NPARAM]
    float *mlp_grad = nullptr;           // gradient + loss [KG_MLP_NPARAM + 1]
    void *mlp_blob = nullptr;            // bf16 image (kg::MlpSmem) for the tensor cores
    void *mlp_w2t = nullptr;             // bf16 W2 transposed, [64][72] (backward)
    long long adam_t = 0;                // Adam steps taken
    long long train_iter = 0;            // minibatches drawn
    double *logf = nullptr, *logt = nullptr;   // per-attempt staging of the sweep log
    int *logn = nullptr, *logoff = nullptr;    // rows of each attempt, their offsets (and the scan's block sums)
    long long log_att_cap = 0;
    double *trainf = nullptr, *traint = nullptr;  // training ring [train_cap][24], [train_cap]
    long long train_cap = 0;
    long long *d_train_head = nullptr;   // rows ever appended
    void *tr_buf = nullptr;              // minibatch work arrays
    long long tr_rows = 0;
    unsigned long long *bmax2 = nullptr; // longest bond squared (binary64 bits), per learned sweep
    double *d_io = nullptr;              // device staging for host-pointer calls
    long long d_io_cap = 0;

    // scratch
    double *scratch = nullptr;   // [3][Mp] doubles + [3][Mp] + [Mp] ints (gather / staging)
    unsigned *flags = nullptr;   // [0] error bits, [1] rebuild request, [3] max list length, [4] blocks done,
                                 // [5] Verlet builds, [6] kernels of captured loops' passes that are no steps,
                                 // [8], [9] RES_BUILT, RES_NEXT
    double *partials = nullptr;  // block partial sums for observables
    int partials_cap = 0;
    double *r2tmp = nullptr;     // per-chain <R^2(n)> partial sums
    long long r2tmp_cap = 0;
    int *hist = nullptr;         // histogram counts
    int hist_cap = 0;
    double *fout = nullptr;      // forces for kg_forces
    double *msd_ref = nullptr;   // [3][Mp] reference positions of kg_msd (+ [3][Mp] re-sort scratch)

    // instrumentation
    long long launches = 0;      // kernels launched since creation
    bool prof_on = false;
    std::vector<cudaEvent_t> ev; // pairs around step-kernel launches
    int ev_used = 0;
    double prof_ms = 0.0;
    long long prof_n = 0;
};

namespace kg {

// a context's own stream waits for the work queued on the default stream so far
void follow_default(kg_ctx *c);
void follow_default_for(kg_ctx *c, const void *out);   // the same before it writes a caller's device memory
// device memory through the context's allocator (zero-filled on the context's stream)
void *dev_alloc(kg_ctx *c, size_t bytes, size_t clear = ~(size_t)0);   // the first `clear` bytes zero
void dev_free(kg_ctx *c, void *p);

constexpr int GRAPH_STEPS = 10;          // MD steps between re-sort tests
constexpr int PERSIST_STEPS = 50;        // MD steps between re-sort tests with KG_FLAG_PERSISTENT
constexpr int RESIDENT_STEPS = 50;       // MD steps per resident launch (KG_FLAG_PERSISTENT, step loop: PERSIST_MAX)
constexpr int PERSIST_MAX = 1000;
constexpr unsigned RESIDENT_SPIN = 1u << 22;  // its barrier polls (0.32 us apart) before ERR_TIMEOUT
constexpr int RS = 8;                    // ints per melt in the DB commit-round array

// A sweep's record of one attempt.  The staleness check of every round reads
// the first 32 bytes only.
struct __align__(16) Attempt {
    int flags;                   // 1: non-empty partner set, 2: accepted, 4: partner drawn, not yet decided
    int c, d;                    // chain of the drawn bond, chain of the chosen partner
    int ver;                     // commits of the melt that the evaluation had seen
    int cell[4];                 // 1.3 sigma cells of the junction monomers (-1: unused)
    int kind, A, B, pA, pB;      // canonical move
    int q;                       // partner bond of chain d
    int n;                       // partners of the drawn bond
    int pad;
    double p, dE;                // learned proposal: probability of the pick, energy change
};

// kg_md.cu
void rebuild_md(kg_ctx *c);                  // conditional on flags[1]
void md_step(kg_ctx *c);                     // one fused force + integrate step (direct launches)
// captured step loop: its start, and the graph of a while node whose body `pass` enqueues on s
void loop_begin(cudaStream_t st, LoopDev *lp, long long steps, int len);
bool capture_loop(cudaStream_t s, cudaGraphExec_t *exec, const std::function<void(cudaGraphConditionalHandle)> &pass);
bool md_loop_steps(kg_ctx *c, int n);        // n steps in one launch of the captured step loop
void set_device_step(kg_ctx *c, long long v);
void forces_eval(kg_ctx *c, int melt, long long step, double *F_dev, double *part_dev, int nblk);
void prof_collect(kg_ctx *c);                // fold recorded event pairs into the totals
void bonded_partners(kg_ctx *c);             // bp from slot_of / comp_of
void scan_counts(kg_ctx *c, const int *count, int *start, int n, int *bsum);   // exclusive scan, start[n] the total
void md_sort(kg_ctx *c);                     // re-sort the state into the last cell order
void md_materialize(kg_ctx *c);              // mixed: x <- xb64 + dlt[cur]
void graphs_reset(kg_ctx *c);                // drop captured step graphs (their arguments changed)

// kg_resident.cu
enum { RES_NONE = 0, RES_WIDE = 1, RES_SMALL = 2, RES_TILED = 3 };
int resident_kind(kg_ctx *c);                // which resident kernel serves the context
cudaError_t resident_launch(kg_ctx *c, int K, int skip_block, unsigned spin);   // K steps in one launch
bool resident_alloc(kg_ctx *c);              // its buffers (none for contexts it does not serve)
cudaError_t resident_reset(kg_ctx *c);
void resident_cell_order(kg_ctx *c);         // clist after builds that used buckets

// kg_step.cu
// the mixed path's fused step kernel; loop, k: its place in a captured step loop
void step_mixed_launch(kg_ctx *c, cudaStream_t st, int cur, LoopDev *loop, int k);
void to_slots(kg_ctx *c, int melt, const double *in_comp, double *out_dev, int dims);
void state_to_slots(kg_ctx *c, int melt, double *x_dev, double *u_dev, int *pid_dev);   // null: not wanted
int forces_blocks(const kg_ctx *c, int melt);

// kg_db.cu
cudaError_t db_sweep(kg_ctx *c, const std::vector<long long> &K, long long *host_stats /*[n_melts][4]*/);
void db_bin(kg_ctx *c, const std::vector<long long> &K);     // attempt offsets + the >= 1.3 sigma grid
void db_finish(kg_ctx *c, long long *host_stats);             // box shifts, chain partners, stats to host
// reset the commit bookkeeping of a sweep (versions, stamps, rounds)
void db_rounds_reset(kg_ctx *c);


// kg_learned.cu
cudaError_t db_sweep_learned(kg_ctx *c, const std::vector<long long> &K, double lambda, long long *host_stats);
bool db_proposal(kg_ctx *c, int melt, int chain, int bond, double lambda, int *h_n, int *h_ints /*[3][48]*/,
                 double *h_f /*[48][24]*/, double *h_s /*[48]*/, double *h_pi /*[48]*/);

// kg_mlp.cu
bool mlp_ensure(kg_ctx *c);                                  // allocate; zero weights on first use
void mlp_set(kg_ctx *c, const double *w_dev);                // FP64 device vector -> master + bf16 image
void mlp_get(kg_ctx *c, double *w_dev);                      // master -> FP64 device vector
void mlp_infer(kg_ctx *c, const double *f_dev, long long n, double *s_dev);
bool mlp_grad(kg_ctx *c, const double *f_dev, const double *t_dev, long long n, double *loss_grad_dev);
bool mlp_train(kg_ctx *c, int iters, int batch, double lr, double *loss_dev);

// kg_obs.cu
constexpr int R2N_SMEM_MAX = 24 * KG_R2N_MAX_CHAIN_LEN;     // bytes of k_r2n_chain's positions
bool r2n_eval(kg_ctx *c, int melt, double *out_dev);          // false: launch failed or N too long
void hist_eval(kg_ctx *c, int melt, int nbins, int *out_dev);
bool msd_reset(kg_ctx *c, int melt);                          // allocates the reference on first use
int msd_blocks(const kg_ctx *c, int melt);
void msd_eval(kg_ctx *c, int melt, double *part_dev);         // block partial sums of |x - ref|^2
void msd_permute(kg_ctx *c, const int *order);                // re-sort (no-op before the first reset)
void sq_eval(kg_ctx *c, int melt, const int *hkl_dev, int nq, long long *part_dev /*[2 nq + 1], zero*/, double *S_dev);
void gr_eval(kg_ctx *c, int melt, int R, double r_max, double dr, int nbins, unsigned long long *hist_dev);
constexpr int GR_BINS_MAX = 2048;

}  // namespace kg
