// Internal declarations shared by the librsot translation units.
//
// Layout in HBM (all device buffers owned by rsot_problem):
//   points  : FP32 translated coordinates, SoA xs[k * nq_pad + q] (k < d),
//             zero-padded to nq_pad (a multiple of the pass-1 point tile);
//             FP64 translated coordinates x64[q * d + k]; masses m_q (FP64)
//             and log2 m_q (FP64).
//   targets : FP64 translated coordinates y64[j * d + k], nu_j, ln nu_j.
//   per evaluation (mixed precision, log2 domain, see rsot_dense.cu):
//             target records        tquad[j]    = (w0,w1,w2,c)
//             target "pair" records TRecPair[g] = (w0a,w0b,w1a,w1b,w2a,w2b,ca,cb)
//             pass-1 partials (M, S) per point and target chunk
//             point records         pquad[q]    = (x0,x1,x2,u) for pass 2
//             pass-2 FP64 partial sums per point chunk and target
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/rsot.h"

namespace rsot {

constexpr double kLog2e = 1.4426950408889634074;
constexpr double kLn2 = 0.69314718055994530942;
constexpr float kPadC = -1.0e30f;            // exponent of a padding target: ex2 -> 0

// Error bits written by kernels into ProblemDev::flags.
enum : int {
    kErrTimeout = 1,        // an mbarrier wait exceeded its iteration limit
    kErrNonfinitePsi = 2,   // psi had a NaN / Inf entry
    kErrBadCell = 4,        // a cell index fell outside the grid (truncated path)
    kErrRange64 = 8,        // the fixed-point passes cannot hold the exponents: FP64 passes instead
};

struct __align__(16) Rec8 {   // 32-byte record: two float4
    float4 a;
    float4 b;
};

// Result block copied back to the host after each evaluation.
struct EvalResult {
    double J;
    double psic;        // psi_0 of the evaluation (the potential centre)
    long long pairs;
    long long empty;
    int flags;
    int gate;           // bit 0: an f16 operand is out of range (both passes take the FP32 kernels)
    unsigned fx_key[3]; // pair skipping (rsot_skip.cuh): largest A_q, B_j, |B_j| as ordered keys
    int fx_F;           // fraction bits of the fixed-point passes (rsot_fx64.cu)
    unsigned ticket;    // blocks of the final kernel that are done
    int ok;             // the last evaluation that ended with the final kernel succeeded
};

struct Grid;  // truncated-path cell grid (rsot_trunc.cu)
struct Rec16; // tensor-core operand record (rsot_tc.cuh)
struct FxRec; // fixed-point operand record (rsot_fx64.cu)

}  // namespace rsot

struct rsot_problem {
    int d = 0;
    int dev = 0;
    int64_t nq = 0, n = 0;
    int64_t nq_pad = 0, n_pad = 0;
    cudaStream_t stream = nullptr;
    double origin[3] = {0, 0, 0};
    double msum = 0.0;          // sum_q m_q
    double hx = 0.0;            // sum_q m_q |x'_q|^2 / 2 (translated coordinates)
    double nu_min = 0.0, nu_max = 0.0;
    double half_ext = 0.0;      // largest half extent of that box along an axis
    double diam2 = 0.0;         // squared diameter of the bounding box of points and targets
    int num_sms = 0;

    // static device data
    float *xs = nullptr;        // [d][nq_pad]
    double *x64 = nullptr;      // [nq][d]
    double *mass = nullptr;     // [nq]
    double *lmass2 = nullptr;   // [nq] log2 m_q (-inf if m_q == 0)
    double *y64 = nullptr;      // [n][d]
    double *nu = nullptr;       // [n]
    double *lnu = nullptr;      // [n] ln nu_j

    // per-evaluation scratch (mixed)
    float4 *tquad = nullptr;        // [n_pad] (w0,w1,w2,c)
    rsot::Rec8 *tpair = nullptr;    // [n_pad / 2]
    float2 *part1 = nullptr;        // [k1][nq_pad]
    float4 *pquad = nullptr;        // [nq_pad] (x0,x1,x2,u)
    double *part2 = nullptr;        // [s2][n_pad]
    double *blockJ = nullptr;       // [nblk_j]
    double *psinu = nullptr;        // [8 nblk_prep] partials of sum psi nu: one per 256 targets or per warp
    int k1 = 0, chunk1 = 0;         // pass-1 target chunks
    int s2 = 0;                     // pass-2 point splits
    int64_t chunk2 = 0;
    char *ms_buf = nullptr;         // skipping mixed passes (rsot_mskip.cu): orders of the rows, partials
    int *ms_perm_q = nullptr, *ms_perm_t = nullptr;
    double *ms_part2 = nullptr;     // [ms_s2][n_pad]
    int ms_s2 = 0;
    int64_t ms_chunk2 = 0;
    bool cent_now = false;          // this evaluation also forms the centroids' sums
    int cent_tpp = 0, cent_s2 = 0;  // target pairs per thread, point splits of that pass
    int64_t cent_chunk = 0;
    double *cent_part = nullptr;    // [cent_s2][d + 2][n_pad]
    char *plan_dev = nullptr;       // outputs of maps and centroids for host memory (rsot_api.cu)
    char *plan_host = nullptr;      // pinned
    size_t plan_dev_bytes = 0, plan_host_bytes = 0;
    int s2_eval = 0;                // outside the solver (dense_alloc)
    int64_t chunk2_eval = 0;
    int nblk_comb = 0, nblk_prep = 0;
    int per_comb = 1, per_prep = 1; // partials per 256 points / targets: 1, or 8 (one per warp)
    // tensor-core form of the pair arithmetic (rsot_tc.cuh)
    rsot::Rec16 *trec = nullptr;    // [n_pad] target operand records
    rsot::Rec16 *prec16 = nullptr;  // [nq_pad] point operand records (static)
    float *pu = nullptr;            // [nq_pad] pass-2 shifts u_q = log2 m_q - R_q
    float tc_P = 1.0f;              // point coordinate scale (power of two)
    int pair_kernel = 2;            // 0: FP32 passes, 1: tensor-core passes (FP32 fallback by
                                    // gate), 2: tensor-core passes when m_max nu_max <= kTcAuto
    double m_max = 0.0;             // max_q m_q
    // estimated L1 norm of the tensor-core rounding noise of a gradient,
    // 1.4e-5 sqrt(m_max) sum_j sqrt(nu_j) (see kTcAuto); solvers take the FP32
    // kernels once the gradient is within kTcNoiseFactor of it
    double tc_noise_l1 = 0.0;
    int pair_fp32_now = 0;          // set by a solver: this evaluation takes the FP32 kernels
    int in_solve = 0;               // set while rsot_solve runs on this handle
    int k1_tc = 0, chunk1_tc = 0;   // pass-1 target chunks of the tensor-core launch
    int s2_tc = 0;                  // pass-2 point splits of the tensor-core launch
    int64_t chunk2_tc = 0;
    // FP64 path scratch
    double *a64 = nullptr;          // [n_pad]   psi_j/eps + ln nu_j
    double *prec64 = nullptr;       // [nq_pad][4] (x0,x1,x2,u)
    int s2_64 = 0;
    int64_t chunk2_64 = 0;
    double *part2_64 = nullptr;     // [s2_64][n_pad]
    // pair skipping of the dense FP64 and compensated passes (rsot_skip.cu): one
    // allocation on first use
    void *sk_buf = nullptr;
    float *sk_part = nullptr;                              // largest exponents per target chunk
    float4 *sk_ptrow = nullptr, *sk_ptcol = nullptr, *sk_tgrow = nullptr;   // FP32 records
    float *sk_ptA = nullptr, *sk_tgB = nullptr;            // values of the ball test
    int *sk_perm = nullptr;                                // order of the target rows
    int sk_pp = 0, sk_k = 0;
    int *sk_perm_q = nullptr;       // order of the point pairs (large problems)
    int64_t sk_chunk = 0;
    // fixed-point passes of the dense FP64 path (rsot_fx64.cu): one allocation on first use
    void *fx_buf = nullptr;
    rsot::FxRec *fx_prec = nullptr, *fx_trec = nullptr;   // integer operands of points, targets
    int *fx_ptshift = nullptr, *fx_tgshift = nullptr;     // integral row shifts
    double *fx_tgscale = nullptr;                         // 2^(fraction of B_j)
    double *fx_tab = nullptr;                             // 2^(-i/2048)
    double *fx_part1 = nullptr, *fx_part2 = nullptr;      // row sums per column chunk
    int fx_k1 = 0, fx_s2 = 0;
    int64_t fx_chunk1 = 0, fx_chunk2 = 0;
    // compensated dense evaluation outside the solver (rsot_cx.cu): one allocation on first use
    void *cx_buf = nullptr, *cx_prec = nullptr, *cx_trec = nullptr;
    double *cx_part1 = nullptr, *cx_part2 = nullptr;
    float *cx_shift = nullptr;
    int cx_s2 = 0;
    int64_t cx_chunk2 = 0;
    // compensated path scratch (rsot_df.cu), allocated on first use
    void *df_prec = nullptr;        // [nq_pad] point head/tail records (64 B)
    void *df_trec = nullptr;        // [n_pad] target head/tail records (64 B)
    double *df_part2 = nullptr;     // [df_s2][n_pad] pass-2 partials
    int df_s2 = 0;
    // truncated compensated passes: targets in the Morton order of the cell list,
    // blocks classified by balls (rsot_df.cu)
    double *df_beta_s = nullptr;    // [n_pad] beta in sorted order (per evaluation)
    float *df_beta_sf = nullptr;    // [n_pad] nb_j = b_j - 2k beta_j in FP32, sorted (per evaluation)
    float *df_alpha_f = nullptr;    // [nq_pad] A_q = k|x'_q|^2 - 2k alpha_q in FP32 (per evaluation)
    float4 *df_pb64 = nullptr;      // [nq_pad / 64] balls of 64 caller-order points (once)
    float4 *df_pb8 = nullptr;       // [nq_pad / 8] balls of 8 caller-order points (once)
    float2 *df_pa64 = nullptr, *df_pa8 = nullptr;    // alpha ranges of those point blocks
    float2 *df_tbe64 = nullptr, *df_tbe8 = nullptr;  // beta ranges of 64 / 8 sorted targets

    // truncation cutoffs per pair, c(x_q, y_j) < alpha_q + beta_j (rsot_cutoff.cu)
    int *nn = nullptr;              // [nq] nearest target of each point (once per problem)
    double *nn_c = nullptr;         // [nq] its cost
    double *alpha = nullptr;        // [nq_pad] per evaluation (-inf for padding)
    double *beta = nullptr;         // [n_pad]  per evaluation (-inf for padding)
    int cut_anchored = 0;           // alpha is anchored at the nearest targets (psi-aware)

    // staging for host psi / grad
    double *psi_dev = nullptr;      // [n]
    double *psi_host = nullptr;     // pinned (behind grad_host): a small host potential on its way
    const double *psi_src = nullptr;   // set: the next prep kernel reads psi there and fills psi_dev
    bool borrowed = false;          // mass and nu are the caller's device arrays (not freed)
    double *grad_dev = nullptr;     // [n] gradient of the last evaluation
    double *grad_host = nullptr;    // [n] pinned staging of host gradient outputs
    rsot::EvalResult *res_dev = nullptr;
    rsot::EvalResult *res_host = nullptr;   // pinned
    bool res_clean = false;         // *res_dev is zero (the final kernel leaves it so)
    int final_nonempty = 0;         // truncated: an empty neighbourhood is an error
    double *final_out = nullptr;    // the evaluation's gradient output: the caller's device buffer or
                                    // grad_host, written by the final kernel on success
    int *flags = nullptr;           // device error bits (inside res_dev)

    // per-point log partition of the last evaluation (see rsot_point_log_partition)
    double *lse_buf = nullptr;      // [nq_pad]: R_q (mixed, log2) or L'_q (FP64, natural)
    bool last_dense = true;         // the last evaluation's J, pair and empty-point counts
    double last_J = 0.0;            // (rsot_last_eval; its gradient stays in grad_dev)
    int64_t last_pairs = 0, last_empty = 0;
    int last_kind = -1;             // -1 none, 0 FP64 dense, 1 mixed dense, 2/3 truncated (FP64 /
                                    // mixed cell list), 4/5 compensated
                                    // FP64/mixed, 4/5 compensated dense/truncated
    double last_eps = 0.0;

    // covering cost cache
    double C0 = -1.0;

    // truncated path
    rsot::Grid *grid = nullptr;

    // kernel tracing (rsot_kernel_timing)
    int timing = 0;
    std::vector<cudaEvent_t> tr_events;                 // pool, reused
    std::vector<std::pair<const char *, int>> tr_open;  // (name, first event index)
    int tr_used = 0;
    std::vector<const char *> tr_names;
    std::vector<double> tr_total_ms;
    std::vector<int64_t> tr_count;
};

namespace rsot {

// Choice of the pair kernel of the mixed passes.  Every evaluation whose
// result goes back to the caller takes the FP32 pair arithmetic unless the
// caller asked for the tensor-core form (RSOT_PAIRS_TENSOR).  Inside the
// library's solvers (in_solve), whose stop is certified by compensated or
// FP64 reference evaluations, RSOT_PAIRS_AUTO lets the mixed L-BFGS iterations
// take the tensor-core form while its rounding noise is far below the
// gradient: the exponent's error is within about twice the FP32 chain's
// (measured maxima 5.7 and 2.7 units of 2^-24 times the sum of the magnitudes
// of its terms), random in sign, and a gradient entry sum_q m_q p_qj then
// scatters by ~1.4e-5 sqrt(m_max nu_max); where that scatter is no longer
// small (m_max nu_max > kTcAuto) or the gradient approaches it (pair_fp32_now,
// kTcNoiseFactor) the solver keeps the FP32 kernels, which converge further.
constexpr double kTcAuto = 2e-6;
constexpr double kTcNoiseFactor = 30.0;
inline bool use_tensor_pairs(const rsot_problem *p) {
    if (p->pair_kernel == 1) return true;
    return p->pair_kernel == 2 && p->in_solve && !p->pair_fp32_now && p->m_max * p->nu_max <= kTcAuto;
}

// ---- kernel tracing (rsot_api.cu) -------------------------------------------
// trace_begin/trace_end bracket one launch with events on p->stream when
// tracing is on; trace_collect (after a stream sync) accumulates durations.
void trace_begin(rsot_problem *p, const char *name);
void trace_end(rsot_problem *p);
void trace_collect(rsot_problem *p);

// ---- programmatic dependent launch -----------------------------------------------
// The kernels of one evaluation form a chain of short launches: a kernel that is
// launched with launch_pdl may be scheduled while its predecessor runs and waits
// in pdl_wait() for all of it; each triggers its successor right after its own
// wait, so that at most two kernels are in flight.  Without the attribute both
// calls do nothing.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// at the start of a kernel whose inputs its predecessor writes
__device__ __forceinline__ void pdl_enter() {
    pdl_wait();
    pdl_trigger();
}
template <class... P, class... A>
inline void launch_pdl(bool pdl, void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                       A... args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 1 : 0;
    (void)cudaLaunchKernelEx(&cfg, k, P(args)...);   // cudaGetLastError() reports a failure
}

// A pass overlaps the end of the short kernel before it only where its CTAs and that
// kernel's blocks (`before`) together are at most one per SM: CTAs placed while those
// still hold slots leave some SMs with more of a single wave than others.  Calls without
// and with the overlap, in us: 1,536 x 128 43 -> 40, 1,000 x 8,000 (160 in all) 55 -> 55,
// 1,536 x 8,000 (192) 53 -> 60, 16 x 16,000 (320) 52 -> 110, 61,206 x 5,003 160 -> 225;
// FP64 1,536 x 128 (120) 76 -> 70, 6,000 x 128 (382) 79 -> 103.
// A kernel of few blocks leaves room for a pass of one CTA per SM (3,000 x 4,096: 96 CTAs
// after 64 blocks 56 -> 54, 6,000 x 2,000: 53 -> 49), and a pass of few CTAs (`few`) may
// follow any but the target records' kernel, which lets it start at once: 60,000 x 16 (59
// after 944 blocks) 55 -> 51, 24,576 x 300 (96 after 384) 48 -> 45, centroids 60,000 x 300
// (118 after 944) 73 -> 77, FP64 3,000 x 128 (48 after 144) 74 -> 70.
inline bool overlap_pass(const dim3 &g, int64_t before, int num_sms, int few) {
    const int64_t own = (int64_t)g.x * g.y;
    return own + before <= num_sms || (2 * before <= num_sms && own <= num_sms) || own <= few;
}

// The last kernel of a dense evaluation: gradient and J from the partials, the
// gradient to the caller's buffer on success, the result block to the host.
struct FinalArgs {
    const double *part2;        // [s2][stride] pass-2 partials
    int s2;
    int64_t stride;
    const double *scale;        // per target, or null: grad = scale sum - nu
    const double *blockJ;       // nbj groups of per_j partials of pass 1's J term
    int nbj, per_j;
    int log2_J;                 // they are sum m R_q (log2 domain), else sum m eps L_q
    int per_psi;                // partials of sum psi nu per 256 targets
    int groups = 1;             // threads per target (launch_finalize)
};
cudaError_t launch_finalize(rsot_problem *p, const double *psi_dev, double eps, const FinalArgs &a,
                            double *grad_dev);

// ---- launch helpers implemented in rsot_dense.cu --------------------------
cudaError_t dense_alloc(rsot_problem *p);
void dense_free(rsot_problem *p);
cudaError_t launch_dense_mixed(rsot_problem *p, const double *psi_dev, double eps,
                               double *grad_dev);
cudaError_t launch_dense_fp64(rsot_problem *p, const double *psi_dev, double eps,
                              double *grad_dev);
cudaError_t launch_prep_mixed(rsot_problem *p, const double *psi_dev, double eps);
// threads and blocks of the target records' and of the combining kernels
inline int prep_threads(const rsot_problem *p) { return p->per_prep == 1 ? 256 : 64; }
inline int64_t prep_blocks(const rsot_problem *p) { return p->n_pad / prep_threads(p); }
inline int combine_threads(const rsot_problem *p) { return p->per_comb == 1 ? 256 : 64; }
inline int64_t combine_blocks(const rsot_problem *p) { return p->nq_pad / combine_threads(p); }
// dense FP64 evaluation with fixed-point exponents (rsot_fx64.cu); fx64_ready:
// its buffers exist and the sizes of the exponents allow it
bool fx64_ready(rsot_problem *p, double eps);
// pair skipping (rsot_skip.cu)
bool skip_estimate_fits(const rsot_problem *p, double kappa);
bool skip_ready(rsot_problem *p, double eps);
double skip_t1(const rsot_problem *p);
cudaError_t launch_skip(rsot_problem *p, const double *psi_dev, double eps);
void skip_free(rsot_problem *p);
cudaError_t launch_dense_fx64(rsot_problem *p, const double *psi_dev, double eps, double *grad_dev);
void fx64_free(rsot_problem *p);
// the smallest column split whose CTAs fill the resident slots
int split_for_slots(int64_t units, int64_t tiles, int64_t slots);
// rows 0 .. n (row j at pos[j step][d]) by the cells of a grid along the Morton curve, those of
// a cell in their own order, then n .. n_pad as they are; scratch: cell_order_scratch(n) bytes
size_t cell_order_scratch(int64_t n);
cudaError_t cell_order(rsot_problem *p, const double *pos, int64_t n, int64_t n_pad, int *perm, void *scratch,
                       int step = 1);
// dense mixed passes without the pairs that cannot matter (rsot_mskip.cu)
int mskip_ready(rsot_problem *p, double eps);   // bit 0: pass 1, bit 1: pass 2
void mskip_lse(rsot_problem *p, double eps);
void mskip_grad(rsot_problem *p, double eps);
void mskip_free(rsot_problem *p);
// compensated dense evaluation outside the solver (rsot_cx.cu)
bool cx_ready(rsot_problem *p, double eps);
cudaError_t launch_compensated_cx(rsot_problem *p, const double *psi_dev, double eps, double *grad_dev);
void cx_free(rsot_problem *p);
cudaError_t launch_trunc_fp64(rsot_problem *p, const double *psi_dev, double eps, double *grad_dev);
cudaError_t launch_covering_cost(rsot_problem *p, double *C0_dev);
cudaError_t launch_psi_stats(rsot_problem *p, const double *psi_dev, double *out3_dev);
cudaError_t launch_point_L(rsot_problem *p, double *L_dev);
// Copy an evaluation's gradient src -> dst only when the result block reports
// success (no error bit, finite J, and with require_nonempty no empty point).
cudaError_t launch_commit_grad(const double *src, double *dst, int64_t n,
                               const EvalResult *res, int require_nonempty, cudaStream_t st);
cudaError_t launch_softmax_refine(rsot_problem *p, const double *psi_dev, double eps, int64_t nf,
                                  const double *yf_dev, double *out_dev);

// ---- truncation cutoffs (rsot_cutoff.cu): fill p->alpha / p->beta
cudaError_t cutoffs_uniform(rsot_problem *p, double C);
cudaError_t cutoffs_separable(rsot_problem *p, const double *psi_dev, double eps, double tail);
void cutoff_free(rsot_problem *p);
// ln sum_q m_q exp(-L_q) from natural per-point log partitions on the device
cudaError_t launch_log_D(rsot_problem *p, const double *L_dev, double *lnD);

// ---- compensated path (rsot_df.cu): dense, or truncated by p->alpha / p->beta
cudaError_t launch_compensated(rsot_problem *p, const double *psi_dev, double eps, bool trunc,
                               double *grad_dev);
void compensated_free(rsot_problem *p);
// Bound of ||g - grad J||_1 / sum_q m_q for a compensated gradient g (rsot_df.cu)
constexpr double kCompGradRel = 6.5e-7;

// ---- transport maps and centroids (rsot_maps.cu), after a dense mixed evaluation
cudaError_t launch_maps(rsot_problem *p, double eps, double *T_dev, int64_t *j_dev);
cudaError_t cent_ready(rsot_problem *p);   // before an evaluation with cent_now
cudaError_t launch_centroids(rsot_problem *p, double *T_dev, double *mass_dev);

// ---- truncated path (rsot_trunc.cu) ----------------------------------------
// truncated by the cutoffs in p->alpha / p->beta
cudaError_t trunc_eval(rsot_problem *p, const double *psi_dev, double eps, int mixed,
                       double *grad_dev);
void trunc_free(rsot_problem *p);
cudaError_t trunc_point_L(rsot_problem *p, double *L_dev);
// the cell list's target order for the compensated passes (grid built on first
// use): perm (sorted -> caller index, -1 for padding), sorted FP64 coordinates
// [n_pad][d], balls of 8 and of 64 sorted targets [n_pad / 8], [n_pad / 64]
struct SortedTargets {
    const int *perm = nullptr;
    const double *y64 = nullptr;
    const float4 *ball8 = nullptr, *ball64 = nullptr;
};
cudaError_t trunc_sorted_targets(rsot_problem *p, SortedTargets *out);
// block data of the truncated block-skip passes from p->alpha / p->beta
// (rsot_df.cu): df_beta_s, df_alpha_f (A_q), balls and ranges of point and
// target blocks; T receives the sorted-target view
cudaError_t trunc_block_setup(rsot_problem *p, double eps, SortedTargets *T);

// ---- device helpers ----------------------------------------------------------
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float max3f(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// 2^k for an integer-valued float k <= 0 (exact; 0 below the normal range).
__device__ __forceinline__ float pow2_int_f(float k) {
    return k < -126.0f ? 0.0f : __int_as_float(((int)k + 127) << 23);
}
__device__ __forceinline__ double pow2_int_d(float k) {
    return k < -1022.0f ? 0.0 : __longlong_as_double((long long)((int)k + 1023) << 52);
}

// floats as unsigned keys in the same order (for atomicMax); 0 is below every float
__device__ __forceinline__ unsigned ordered_key(float f) {
    const unsigned b = __float_as_uint(f);
    return b & 0x80000000u ? ~b : b | 0x80000000u;
}
__device__ __forceinline__ float from_key(unsigned k) {
    return __uint_as_float(k & 0x80000000u ? k & 0x7fffffffu : ~k);
}

// ---- mbarrier + bulk-copy (TMA) wrappers ------------------------------------
constexpr long long kWaitLimit = 1ll << 24;   // bounded spin: ~seconds at most

__device__ __forceinline__ unsigned smem_u32(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
}
__device__ __forceinline__ void fence_barrier_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_g2s(void *smem, const void *gmem, unsigned bytes,
                                         uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(smem_u32(smem)),
        "l"(gmem), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, unsigned phase) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(phase)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Bounded wait; false when the limit is reached (the caller records an error).
__device__ __forceinline__ bool mbar_wait_n(uint64_t *bar, unsigned phase, long long limit) {
    for (long long i = 0; i < limit; ++i)
        if (mbar_try_wait(bar, phase)) return true;
    return false;
}
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned phase) {
    return mbar_wait_n(bar, phase, kWaitLimit);
}

// Classification of a block pair for the truncated passes: balls a, b (centre,
// radius; radius < 0: no member) of the two blocks and the (min, max) of their
// members' cutoff terms ra, rb (alpha of points, beta of targets; the pair is
// kept when |x - y|^2 / 2 < alpha_q + beta_j).  0: every pair outside, 1: every
// pair inside, 2: boundary (each pair tested).  The radii are widened /
// narrowed by 1e-4 relative, far more than the rounding of the pairwise tests.
// square root on the SFU (sqrt.approx, relative error about 2^-23): far inside
// the classification margins of 1e-4 relative
__device__ __forceinline__ float sqrt_sfu(float x) {
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ int tp_class(float4 a, float4 b, float2 ra, float2 rb) {
    if (a.w < 0.f || b.w < 0.f) return 0;
    const float dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z;
    const float dist = sqrt_sfu(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
    const float Rout = sqrt_sfu(fmaxf(0.f, 2.f * (ra.y + rb.y))) * (1.0f + 1e-4f) + 1e-6f;
    if (dist - a.w - b.w >= Rout) return 0;
    const float Rin = sqrt_sfu(fmaxf(0.f, 2.f * (ra.x + rb.x))) * (1.0f - 1e-4f) - 1e-6f;
    if (dist + a.w + b.w < Rin) return 1;
    return 2;
}

// Block-wide FP64 sum (blockDim.x a multiple of 32, <= 1024); result in thread 0.
__device__ __forceinline__ double block_sum_d(double v, double *sh /* >= 32 */) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) sh[w] = v;
    __syncthreads();
    double r = 0.0;
    if (w == 0) {
        r = (l < (int)(blockDim.x >> 5)) ? sh[l] : 0.0;
        for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
    }
    __syncthreads();
    return r;
}
// block_sum_d of two values at once (thread 0 has the sums)
__device__ __forceinline__ void block_sum2_d(double &a, double &b, double *sh /* >= 64 */) {
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
        sh[threadIdx.x >> 5] = a;
        sh[32 + (threadIdx.x >> 5)] = b;
    }
    __syncthreads();
    const int nw = (blockDim.x + 31) / 32;
    if (threadIdx.x < 32) {
        a = (int)threadIdx.x < nw ? sh[threadIdx.x] : 0.0;
        b = (int)threadIdx.x < nw ? sh[32 + threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_down_sync(0xffffffffu, a, o);
            b += __shfl_down_sync(0xffffffffu, b, o);
        }
    }
}

// Partial sums of v: one per block of 256 threads, or one per warp in smaller
// blocks (kSmall), which final_term() adds in the order of block_sum_d -- the
// same bits either way.  Smaller blocks spread the FP64 work of few targets or
// points over more SMs: 16 blocks of 256 threads kept 16 SMs' two FP64 lanes busy
// for 7 us.
constexpr int kSmall = 64;
inline unsigned small_threads(int64_t rows, int num_sms) { return rows / 256 < 2 * num_sms ? kSmall : 256; }
__device__ __forceinline__ void store_partial(double v, double *__restrict__ out) {
    if (blockDim.x == 256) {
        __shared__ double sh[32];
        const double s = block_sum_d(v, sh);
        if (threadIdx.x == 0) out[blockIdx.x] = s;
    } else {
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) out[blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)] = v;
    }
}

}  // namespace rsot
