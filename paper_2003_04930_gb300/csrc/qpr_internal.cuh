// Internal declarations shared by the solver's translation units.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <stdint.h>

#include <stdio.h>
#include <stdlib.h>

#include <string>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "qpr.h"

namespace qpr {

// A named NVTX range for the length of a scope: every C-ABI call and every
// block of steps shows up on an Nsight timeline (a no-op when no tool is
// attached).
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};

// QPR_LOG=1 in the environment: one line per solve on stderr.
inline bool log_enabled() {
    static const bool on = [] {
        const char *v = getenv("QPR_LOG");
        return v && v[0] && v[0] != '0';
    }();
    return on;
}


struct HostOps;

// Device control block. The host writes tol, dt and max_steps before a
// solve; the kernels read them (so a captured CUDA graph serves every dt)
// and write the stop decision and the residual. Kernels of a step read
// `done` on entry and return at once when it is set.
struct Ctl {
    int done;           // 1: every later kernel returns immediately
    int status;         // kCtlRunning / kCtlConverged / kCtlMaxSteps / kCtlNonFinite
    long long step;     // completed RK4 steps in this solve
    long long max_steps;
    double tol;         // stop when ||f(y_n)||_F < tol (0: never)
    double dt;
    double scale;       // 1 / Re tr(y) of the current step (set by the stage-1 gain kernel)
    double trace;       // Re tr(y) of the current step
    double resid;       // residual of step index `resid_step`
    long long resid_step;
    double resid_exact; // exact FP64 residual of the last reference refresh (mixed form)
    long long resid_exact_step;
    int err_timeout;    // a bounded device-side wait gave up
    int ticket;         // CTAs that finished the current ticketed epilogue (RKF45 stage 6)
    // FP32 forms of dt for the mixed form's delta stages, written by its
    // refresh: dtf = fl(dt), dt = dtf + dtl as a float-float pair, dt3 =
    // fl(dt / 3)
    float dtf, dtl, dt3, pad2_;
    // grid barrier of the persistent column-block kernel: arrivals, generation
    unsigned gb_count, gb_gen;
    // testing only: arrivals a grid barrier waits for beyond its grid (0, or 1
    // to make every barrier wait run out; qpr_options.test_fault)
    unsigned gb_extra, pad3_;
    // RKF45 (qpr_rkf45): the step of the next attempt and its largest value,
    // the tolerance Tol of Eq. S13, the integrated time and its end (0: none),
    // the discrepancy |z - y| of the last attempt, the rejected attempts, the
    // delta pair holding the current state (0: D, Dlo; 1: D1, Dlo1), the
    // order of the solution an accepted attempt keeps (4: y of Eq. S11, 5: z
    // of Eq. S12) and the step as a float-float pair (hf + hl) for the delta
    // stages
    double rk_h, rk_hmax, rk_tol, rk_t, rk_tend, rk_err;
    long long rk_rejected;
    int rk_cur, rk_order;
    float rk_hf, rk_hl;
};

// kCtlCandidate: the mixed form's FP32-accurate residual estimate passed;
// the host confirms it with an exact FP64 refresh.
// kCtlTimeReached: an RKF45 trajectory reached its end time.
enum { kCtlRunning = 0, kCtlConverged = 1, kCtlMaxSteps = 2, kCtlNonFinite = 3, kCtlCandidate = 4,
       kCtlTimeReached = 5 };

// Operators on the device (built once by qpr_create).
struct DevOps {
    int n;                // nodes
    int np;               // padded edge of every N x N plane (multiple of kPadFp64)
    double alpha, omega;
    int dangling;         // QPR_DANGLING_F / QPR_DANGLING_UNIFORM
    const double *H;      // np x np row-major, zero padding
    const int *h_ptr;     // CSR of H (same values; zeros skipped): n + 1 row pointers
    const int *h_col;
    const double *h_val;
    const float *h_val32; // the same values rounded to FP32 (mixed form)
    // rows of H cut into segments of at most 32 nonzeros (mixed form):
    // segments of row i are seg[rowseg[i] .. rowseg[i+1]), each {q0, q1}
    // into h_col / h_val; rowseg has np + 1 entries (empty for padding)
    const int *rowseg;
    const int2 *seg;
    const int *s_ptr;     // CSR of S restricted to columns with out-links: n + 1 row pointers
    const int *s_col;
    const double *s_val;  // A_ij / outDeg(j)
    const unsigned char *dang;  // n flags: column j has no out-links
    const double *c;      // np column sums of G (0 on padding)
    const float *c32;     // the same in FP32 (mixed form)
    // FP32 copies for the mixed form's delta stages (no FP64 instruction in
    // a delta stage): S values, alpha, 1 - alpha, omega, 1 / (n - 1), 1 / n
    const float *s_val32;
    float alpha32, oma32, omega32, inv_nm1_32, inv_n32;
    // column-block form of the sparse mixed stage (plan of ColPlan; 0 splits:
    // not used): the entries of H as (column, FP32 value bits), per bundle
    // interleaved and zero-padded; per row split its entry range {first
    // (even), end} and bundle range; bundle descriptors (2 int4 each); per
    // (split, warp) the first bundle
    const int2 *col_kh;
    const int *col_q;      // 2 per split
    const int *col_sb;     // splits + 1: bundles of split r are [col_sb[r], col_sb[r + 1])
    const int4 *col_pieces;
    const int *col_wb;     // splits * 16 + 1, absolute bundle indices
    int col_splits;
    int col_smem;          // dynamic shared memory of the SpMM kernel
    int col_p_off;         // byte offset of the staged bundles in it
    int col_sp_off;        // byte offset of the staged diagonal (np floats) in it
    int col_gather;        // 1: the gather form (the SpMM reads delta from L2; plan of ColPlan, gather)
    // rows cut into parts (kPartMax): per split the cut range [col_cutb[k], col_cutb[k + 1]) of col_cut; the partial
    // slots at byte col_part_off of the SpMM's shared memory
    const int4 *col_cut;
    const int *col_cutb;
    int col_part_off;
    int col_epi_off;       // persistent form: byte offset of the epilogue buffers (0: over the column block)
    int col_psmem;         // persistent form: dynamic shared memory of its launch
    int col_gain_ctas;     // two-launch forms: leading CTAs of the SpMM grid that form the gain instead
    int col_launch_smem;   // two-launch forms: dynamic shared memory of the SpMM launch (>= np floats)
};

// RK4 work buffers. Every state buffer holds two np x np FP64 planes,
// real part first, then imaginary part.
struct Work {
    double *y;            // state at the start of a step (unnormalised)
    double *z;            // RK4 accumulator
    double *ya, *yb;      // stage inputs (ping-pong)
    double *g;            // gain G p of the current stage, np entries
    double *partials;     // one residual partial per stage-kernel CTA
    int2 *pairs;          // tile pairs (I, J), I <= J, off-diagonal first
    int4 *pairs64;        // the same as {I, J, index in pairs, 0}, most work first (sparse stage)
    int npairs;
    int tiles;            // np / kTileFp64
    Ctl *ctl;
};

// Buffers of the mixed-precision form (stage_mixed.cu). The state is
// y = R + delta: FP64 R = y / tr(y) at the last refresh and F = f(R); the
// delta since that refresh as a float-float pair of FP32 planes, D (high
// part, the FP32 delta the stages read) and Dlo (low part). FP32 (two np x np
// planes each): F32 = fl(F), dt F = Ghi + Glo (float-float) and the stage
// inputs da/db (the nested RK4 form keeps no running stage sum).
struct TcMaps;
struct DigitWork;
struct DigitMaps;
struct MixedWork {
    double *R, *F;
    float *F32, *D, *Dlo, *da, *db, *Ghi, *Glo;
    float *g;             // gain of the stage delta, np
    float *pv;            // np: diagonal of the next stage input (written by every epilogue, zeroed by a refresh)
    double *g64;          // FP64 gain used by the refresh, np
    double *partials;     // exact residual partials of the refresh
    float *partials32;    // residual-estimate partials of the stage-1 kernel
    int2 *pairs;          // 32 x 32 tile pairs (tile-pair stage kernel)
    int4 *pairs64;        // the same for the refresh (Work::pairs64)
    int4 *epi_pairs;      // the same pairs in the column-block epilogues' CTA order: {I, J, index in pairs, 0}
    int npairs;
    int tiles;
    Ctl *ctl;
    int nstage_partials;  // residual partials the stage-1 kernel writes
    // dense backend (tcgen05): the BF16 split planes [3 levels][2 planes: Re,
    // -Im][np][np] of the stage-1, stage-2 and stage-3 inputs (D, da, db);
    // null for the sparse backend
    __nv_bfloat16 *splitD, *splitA, *splitB;
    const TcMaps *maps;   // host pointer, used only by the launch code
    // dense backend, host pointers: the refresh evaluates f(R) with the exact
    // digit products where there is a plan (null: the sparse FP64 stage)
    const DigitWork *digits;
    const DigitMaps *digitmaps;
    // column-block form of the sparse backend and dense backend: X = H delta
    // (2 planes); column-block form: the TMA maps of the stage inputs D, da, db (host pointer; null: tile-pair
    // kernel)
    float *X;
    const struct ColMaps *cmaps;
    // RKF45 in the column-block form (null until the first qpr_rkf45 call):
    // the second delta pair (D1, Dlo1; the controller's rk_cur selects the
    // current one), the running sum of the step's power terms (acc, 2
    // planes), the low part of F as a float-float pair with F32 (Flo, 2
    // planes), and the compact diagonals of D and D1 (pvd, 2 np)
    float *D1, *Dlo1, *acc, *Flo, *pvd;
};

// TMA descriptors of the stage inputs D, da, db for the column-block SpMM:
// each pair of planes seen as 2 np rows of np FP32, boxes of 8 x 256.
struct ColMaps {
    CUtensorMap d[3];
    CUtensorMap d1;  // D1 of the RKF45 form (encoded by its first call)
};

constexpr int kTileTc = 128;

// TMA descriptors of the dense mixed stage: H split planes [3][np][np] and
// the three delta-split buffers.
struct TcMaps {
    CUtensorMap h;
    CUtensorMap d[3];
    int levels;  // leading planes of H that are not zero
    int sms;
};

constexpr int kTileFp64 = 32;
constexpr int kPadFp64 = 32;

// ---- kernels (aux_kernels.cu) ----
// Hermitise an interleaved complex128 n x n matrix into two np x np planes.
void launch_import(const double *rho_il, int n, int np, double *planes, cudaStream_t s);
// planes * ctl->scale (use_scale) -> interleaved complex128 n x n.
void launch_export(const double *planes, int n, int np, const Ctl *ctl, int use_scale,
                   double *rho_il, cudaStream_t s);
// p[i] = Re rho_ii of an interleaved complex128 matrix.
void launch_diag(const double *rho_il, int n, double *p, cudaStream_t s);
// g = G p_s for stage `stage` (0: plain right-hand side, 1..4: RK4 stages).
void launch_gain(int stage, const DevOps &ops, const double *yin, const Work &w, cudaStream_t s);

// ---- FP64 tile-pair stage kernel (stage_fp64.cu) ----
// stage 0: out = f(yin) into w.z, residual partials.
// stage 1..4: one classical RK4 stage with the fused update.
void launch_stage_fp64(int stage, const DevOps &ops, const Work &w, cudaStream_t s);
// Opt in to the kernel's dynamic shared memory on the current device.
cudaError_t init_stage_fp64();

// ---- FP64 dense stage on the tensor cores (stage_digits.cu), same contract ----
// Plan: b bits per digit, s digits of every row of Y, sh of H; erow: per row
// of H the binary exponent of its first digit's unit.
struct HostOps;
struct DigitPlan {
    int b = 0, s = 0, sh = 0;
    std::vector<int> erow;
};
struct DigitWork {
    int b, s, sh;
    int ring_a, ring_b;   // pipeline depths: digit planes of H, blocks of Y
    int gain_ctas;        // leading CTAs of the product launch that form the gain beside their tile
    unsigned tmem_cols;
    int epi_smem;         // dynamic shared memory of the epilogue
    void *yd;             // FP16 digits of the stage input [s][2 planes][np][np]
    int *ecol;            // [2 planes][np]: the exponent of the first digit's unit of a row of Y
    int *erow;            // np
    double *x;            // [H Re Y ; -H Im Y] without the diagonal of Y, 2 planes
    const void *hd;       // digit planes of H
    const double *h;      // H, np x np (several digits)
    int unit;             // one digit: H is the digits times 2^unit
    double *diag;         // the diagonal of the stage input, np
    const double *hc;     // omega / 2 c, np
};
struct DigitMaps {
    CUtensorMap h, y;
};
// False if no digit width keeps the sums exact (stage_fp64.cu serves then).
bool plan_digits(const HostOps &h, DigitPlan &p);
// FP16 values of the digit planes, doubles of x; ints: 3 np.
size_t digits_half_count(const DigitPlan &p, int np);
size_t digits_double_count(const DigitPlan &p, int np);
cudaError_t init_digits(const DevOps &ops, const DigitPlan &p, int sms, void *halves, int *ints, double *x, DigitWork *dw,
                        DigitMaps *maps);
// The whole stage: digits of its input, product (with the gain and, at stage
// 2, the stop decision), epilogue.
void launch_stage_digits(int stage, const DevOps &ops, const Work &w, const DigitWork &d, const DigitMaps &m,
                         cudaStream_t s);
constexpr int kDigitLaunches = 3;

// ---- sparse (CSR H) FP64 stage kernel (stage_sparse.cu), same contract; it
// forms the gain itself ----
// The tile pairs of an np x np problem, the ones with most nonzeros first.
std::vector<int4> pairs_by_work(const HostOps &h, int np);
void launch_stage_sparse(int stage, const DevOps &ops, const Work &w, cudaStream_t s);
cudaError_t init_stage_sparse();

// ---- FP64 RK4 of a small problem, one cluster, many steps a launch (stage_small.cu) ----
// Up to `limit` steps from the state in w.y, or until the stop rule sets
// ctl->done; nnz: the entries of H. One launch is at most kSmallSteps steps
// (40 ms at the largest N). The line at 44: the last size with an octet of
// lanes per element in one cluster's warps; at 45 the eight launches take 366
// us a step, at 44 this form 39.
constexpr int kSmallMaxN = 44;
constexpr int kSmallSteps = 1024;
cudaError_t init_small(int n, int nnz);
cudaError_t launch_small_rk4(const DevOps &ops, const Work &w, int nnz, int limit, cudaStream_t s);

// ---- mixed-precision form (stage_mixed.cu) ----
// Reference refresh: R = y = y / tr(y), F = f(R) exactly (FP64), D = 0, exact
// residual and stop decision.
void launch_mixed_refresh(const DevOps &ops, const MixedWork &w, cudaStream_t s);
// One RK4 stage. Column-block and dense forms: parts & 1 launches the product
// (its leading CTAs form the gain), parts & 2 the epilogue (3 = both, in that
// order); tile-pair form: parts & 2 the stage kernel, which does everything.
// serial (profiling): no programmatic dependent launch.
void launch_mixed_stage(int stage, const DevOps &ops, const MixedWork &w, cudaStream_t s, int parts = 3,
                        bool serial = false);
// Opt in to the dynamic shared memory of the sparse mixed stage kernels.
cudaError_t init_stage_mixed();
// Dense backend of the mixed form (stage_mixed_tc.cu).
cudaError_t init_mixed_tc();
bool make_tc_maps(const DevOps &ops, const __nv_bfloat16 *hsplit, int levels, int sms,
                  const __nv_bfloat16 *const dsplit[3], TcMaps *maps);
// X = H delta (with the gain and, at stage 2, the stop decision in its leading CTAs).
void launch_mixed_tc_product(int stage, const DevOps &ops, const MixedWork &w, const TcMaps &m, cudaStream_t s, bool pdl);
// The epilogue of the forms that write X (the column forms and the dense one).
void launch_x_epilogue(int stage, const DevOps &ops, const MixedWork &w, cudaStream_t s, bool pdl);
// Column-block form of the sparse mixed stage (stage_cols.cu): per stage a
// column-block SpMM X = H delta from TMA-staged columns, then the tile-pair
// epilogue. Used where its staged operands fit (np <= kColMaxNp and a plan).
constexpr int kColMaxNp = 1536;
// Complex columns per block of the whole-block and of the gather SpMM.
constexpr int kColWidth = 16;
constexpr int kColGatherWidth = 32;
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder();
bool make_col_maps(const DevOps &ops, const float *const din[3], ColMaps *maps);
// Host plan of the column-block SpMM (device copies go to DevOps col_*).
struct ColPlan {
    int splits = 0;
    int smem = 0;                 // dynamic shared memory per CTA
    int p_off = 0;                // byte offset of the staged bundles
    int sp_off = 0;               // byte offset of the staged diagonal
    std::vector<int2> kh;         // entries of the bundles, interleaved and padded
    std::vector<int> q;           // 2 per split
    std::vector<int> sb;          // splits + 1
    std::vector<int4> pieces;     // 2 per bundle
    std::vector<int> wb;          // splits * 16 + 1
    std::vector<int4> cuts;       // rows cut into parts: {row, first partial slot, parts, 0}
    std::vector<int> cutb;        // splits + 1: the cuts of split r are [cutb[r], cutb[r + 1])
    int part_off = 0;             // byte offset of the partial slots in the SpMM's shared memory
};
// Plans the column-block form of an np x np problem on `device`; false if
// its staged operands do not fit one CTA's shared memory. Row splits: the
// fewest from min_splits up that fit (0: enough CTAs for every SM when the
// problem runs alone). A row's product does not depend on the plan (its
// group sums its entries in order; zero padding never changes a sum that
// starts at +0), so every plan gives bitwise the same X.
// gather: the plan of the gather form (no staged column block, any np; row
// splits from enough CTAs for every SM several times over).
bool plan_columns(const HostOps &h, int np, int device, ColPlan &plan, int min_splits = 0, bool gather = false);
cudaError_t set_gather_smem(int bytes);
// Opt in to `bytes` of dynamic shared memory for the SpMM kernels.
cudaError_t set_cols_smem(int bytes);
void launch_cols_stage(int stage, const DevOps &ops, const MixedWork &w, cudaStream_t s, int parts = 3,
                       bool serial = false);
// RKF45 in the column-block form (stage_rkf.cu). One attempt is six
// stages, each the SpMM (its leading CTAs form the gain) and the epilogue;
// stage 6 ends with the step-size controller. The refresh folds the current delta into R and
// recomputes F = f(R) exactly, as the RK4 refresh does.
constexpr int kRkfStages = 6;
constexpr int kRkfLaunchesPerAttempt = 2 * kRkfStages;
bool make_rkf_map(const DevOps &ops, const float *d1, ColMaps *maps);
void launch_rkf_stage(int stage, const DevOps &ops, const MixedWork &w, cudaStream_t s);
void launch_rkf_refresh(const DevOps &ops, const MixedWork &w, cudaStream_t s);
constexpr int kRkfLaunchesPerRefresh = 4;
cudaError_t init_rkf(int spmm_smem, bool gather);

// Persistent form (stage_persist.cu): one cooperative launch runs up to
// `steps` RK4 steps of the column-block form, grid barriers between the
// phases. persist_grid: CTAs of that launch for an np x np problem with the
// given plan on `device` (0: the form does not apply).
// On success also the launch's dynamic shared memory and the offset of the
// epilogue buffers in it.
int persist_grid(int np, int splits, int smem, int device, int *persist_smem, int *epi_off);
cudaError_t set_persist_smem(int bytes);
cudaError_t launch_cols_block(const DevOps &ops, const MixedWork &w, int steps, int grid, cudaStream_t s);
// Kernel launches per RK4 step and per refresh of the mixed form.
constexpr int kMixedLaunchesPerStep = 4;   // tile-pair sparse kernel (the dense form: a product and an epilogue per stage)
constexpr int kMixedLaunchesPerStepCols = 8;  // column-block form: SpMM (with the gain) and epilogue per stage
inline int mixed_launches_per_refresh(const MixedWork &w) { return w.digits ? 6 : 4; }
// Steady-state solves with adaptive_refresh: the longest window between
// refreshes, in multiples of ref_refresh.
constexpr int kMaxRefreshGrowth = 8;

// ---- classical PageRank and hub classes (pagerank.cu) ----
// CTAs of one power-iteration kernel for n nodes.
int pagerank_grid(int n);
// Power iteration pi <- G pi / sum(pi) from the uniform vector until the L1
// change of an iteration (checked every 8) is below tol or after max_iter
// iterations; pi (normalised) into pi_out_dev (n doubles). scratch: device,
// 2 n + pagerank_grid(n) doubles. Synchronises the stream.
cudaError_t pagerank(const DevOps &ops, double tol, int64_t max_iter, double *scratch, double *pi_out_dev,
                     int64_t *iters, double *delta_out, cudaStream_t s);
// The same for n <= kPrClusterMaxN in one cluster per graph, up to a few
// thousand iterations per launch. scratch: n + kPrState doubles.
// pagerank_in_cluster: whether this form is the faster one for a graph.
constexpr int kPrClusterMaxN = 8192;
constexpr int kPrState = 4;
bool pagerank_in_cluster(const HostOps &h);
cudaError_t pagerank_cluster(const DevOps &ops, double tol, int64_t max_iter, double *scratch, double *pi_out_dev,
                             int64_t *iters, double *delta_out, int64_t *launches, cudaStream_t s);
// A fixed number of power iterations for `count` graphs of at most max_n <=
// kPrClusterMaxN nodes (jobs in device memory), from the uniform vector.
struct PrJob {
    int n, dangling;
    double alpha;
    const int *s_ptr, *s_col;
    const double *s_val;
    const unsigned char *dang;
    double *pi;       // n: the normalised vector (may be null)
    float *feature;   // (float)log(n pi_i) at feature[i * stride] (may be null)
    int stride;
};
cudaError_t pagerank_jobs(const PrJob *jobs, int count, int max_n, int iters, cudaStream_t s);
// classes_dev[i] in {0, 1, 2} (rest, secondary hub, main hub) of the
// probabilities p (device, n doubles) with threshold factor c; counts_dev
// (3 values) receives the class sizes.
cudaError_t hub_classes(const double *p, int n, double c, int *classes_dev, unsigned long long *counts_dev,
                        cudaStream_t s);

// Raise the dynamic shared-memory limit of `kernel` on the current device to
// at least `bytes`; never lower it (contexts with different plans share the
// kernel, and a limit above a launch's request is harmless). Serialised
// over host threads.
cudaError_t raise_smem_limit(const void *kernel, int bytes);
template <typename K>
cudaError_t raise_smem_limit_t(K *kernel, int bytes) {
    return raise_smem_limit(reinterpret_cast<const void *>(kernel), bytes);
}

// ---- host assembly (qpr_api.cu) ----
struct HostOps {
    int64_t n = 0;
    std::vector<double> outdeg;
    std::vector<int64_t> hptr;
    std::vector<int> hcol;
    std::vector<double> hval;
    std::vector<int> sptr, scol;
    std::vector<double> sval;
    std::vector<unsigned char> dang;
};
qpr_status assemble_host(int64_t n, int64_t m, const int64_t *src, const int64_t *dst, const double *w, int h_diag,
                         HostOps &out, std::string &err, bool with_h = true);
// Segments of at most `len` nonzeros of every row of the CSR of H, for np
// rows (rowseg: np + 1 entries, seg: {q0, q1}).
void row_segments(const HostOps &h, int np, int len, std::vector<int> &rowseg, std::vector<int2> &seg);
std::vector<double> column_sums_G(const HostOps &h, double alpha, int np, double *cmax);
// Message returned by qpr_last_error(NULL) on this thread.
void set_create_error(const std::string &msg);
// Opt in to the dynamic shared memory of the batched kernels (batch.cu).
cudaError_t init_batch();
cudaError_t set_bcols_smem(int bytes);
// Resident CTAs per SM of the batched SpMM with `bytes` of dynamic shared memory.
cudaError_t bcols_ctas_per_sm(int bytes, int *ctas);
// Estimate of lambda_max - lambda_min of H (2% margin, at most twice the
// Gershgorin radius): power iteration on the host, or, where spread_on_device
// says so, by spectrum.cu (`raw` its result).
double estimate_spread(const HostOps &h);
bool spread_on_device(const HostOps &h);
// estimate_spread of the problems `which`, on several host threads (false: out of memory).
bool estimate_spreads(const std::vector<HostOps> &h, const std::vector<size_t> &which, std::vector<double> &out);
double bounded_spread(const HostOps &h, double raw);
struct SpectrumJob {
    int n;
    const int *h_ptr, *h_col;
    const double *h_val;
    double *out;
};
// `count` jobs in device memory (or `one`, jobs null), n <= max_n each.
constexpr int kSpectrumMaxN = 8192;
cudaError_t spectral_spread(const SpectrumJob *jobs, int count, int max_n, const SpectrumJob &one, cudaStream_t s);

}  // namespace qpr
