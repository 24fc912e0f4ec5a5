// kernels.h -- launch wrappers of the sm_103a kernels (host-callable).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <vector>

#include "brick.h"
#include "fp_internal.h"

namespace fpk {

struct SampleParams {
    uint64_t seed;
    int32_t n;
    int32_t raw_kind;     // RawKind
    int32_t self_pair;
};

// Let a kernel's launches take up to `most` bytes of dynamic shared memory.  The limit belongs to
// the function, not to a call: `most` is the same for every call of a kernel, so that no host
// thread lowers it between another's call and its launch.
template <typename... A>
inline cudaError_t allow_smem(void (*kernel)(A...), size_t most) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}
// up to all that its static arrays leave of an SM's
template <typename... A>
inline cudaError_t allow_all_smem(void (*kernel)(A...)) {
    cudaFuncAttributes fa;
    int dev = 0, all = 0;
    cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&all, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return e == cudaSuccess ? allow_smem(kernel, (size_t)all - fa.sharedSizeBytes) : e;
}

// Sampler: raw gates of U and V for every pair of the batch (FP64).
cudaError_t launch_sample(const SampleParams &sp, const PairInfo *pairs, int npairs, int max_raw,
                          double2 *raw, cudaStream_t st);
// Haar gates (kernels_haar.cu): raw records (launch_sample's RAW_HAAR4), and the maps of a
// brickwork sweep straight from the sampled gates (launch_brick without raw gates).
cudaError_t launch_haar_raw(const SampleParams &sp, const PairInfo *pairs, int npairs, int max_raw, double2 *raw,
                            cudaStream_t st);
cudaError_t launch_brick_haar_maps(const BrickDev &d, const SampleParams &sp, const PairInfo *pairs, int npairs,
                                   void *maps, bool fp32, cudaStream_t st);
// HEA boundary sweep for boundaries of N = 2L-2 <= 14 bits (kernels_hea.cu): the
// sampled and merged 2x2 slot factors ([pair][qubit][slot][4] of C), then the
// sweep and meet (`states`: one boundary per pair).  hea_shape: window bits and
// threads per CTA of the sweep; false where it does not apply.
cudaError_t launch_hea_slots(const SampleParams &sp, const PairInfo *pairs, int npairs, int L, void *slots, bool fp32,
                             cudaStream_t st);
bool hea_shape(int N, bool fp32, int *win_bits, int *threads);
cudaError_t launch_hea_sweep(const BrickDev &d, const PairInfo *pairs, int npairs, const void *slots, void *states,
                             bool fp32, double err_scale, double *tr, double *kappa, double *err, cudaStream_t st);
// Merged gates: ordered products of raw gates (FP64).
cudaError_t launch_merge(const PairInfo *pairs, int npairs, int max_merged, const DevPlan *plans,
                         const MergeItem *items, const MergeRef *refs, const double2 *raw,
                         double2 *merged, cudaStream_t st);
// Op tables (16 entries per op) in FP64 or FP32.
cudaError_t launch_tables(const PairInfo *pairs, int npairs, int max_ops, const DevPlan *plans,
                          const DevRecipe *recipes, const double2 *merged, void *tables, bool fp32,
                          cudaStream_t st);
// Generic boundary sweep + meet: one cluster of `cs` CTAs (1, 4, 8 or 16) per
// pair at a time, persistent over a ticket queue; `ctas` is a multiple of cs
// and the workspace holds ctas/cs slots of 3 x ws_elems amplitudes.  Writes
// tr[2*i], kappa[i] for pair i of `order`.
cudaError_t launch_sweep_generic(const PairInfo *pairs, const int32_t *order, int count,
                                 const DevPlan *plans, const DevOp *ops, const void *tables,
                                 bool fp32, void *workspace, size_t ws_elems_per_cta, int ctas, int cs,
                                 int *ticket, double err_unit, double *tr, double *kappa, double *err,
                                 cudaStream_t st);
// Lock-step sweep of local-circuit pairs (kernels_step.cu).  Step k of the batch applies
// operation k of both sides of every pair: block i of the launch works on item
// which[step_first[k] + i], on its outputs or groups of outputs ("units")
// (i - first) << log_units and the 2^log_units - 1 after it.
enum StepForm : uint8_t { STEP_IN_PLACE, STEP_1_3, STEP_3_1, STEP_0_4, STEP_4_0, STEP_ANY };
constexpr int kMeetChunk = 14;
struct StepItem {
    uint64_t in, out;        // first amplitudes of the operation's buffers in the workspace
    int64_t table;           // its table
    int32_t op;              // its DevOp
    uint32_t first, units;   // first block of the step's launch; units in all
    uint8_t form, log_units; // StepForm
    uint16_t pad;
};
struct StepPair {
    uint64_t base[2];        // start amplitude of each side
    uint64_t final[2];       // final boundary of each side
    uint32_t first;          // first block of its meet
    uint32_t pad;
};
struct StepBatch {
    const StepItem *items;                 // device
    const uint32_t *which;                 // device
    const StepPair *pairs;                 // device
    const uint32_t *meet_which;            // device
    void *partials;                        // device: 4 doubles per meet block
    std::vector<uint32_t> step_first;      // host: first block of each step, and the end
    uint32_t meet_blocks;
};
cudaError_t launch_steps(const StepBatch &b, const PairInfo *pairs, int npairs, const DevPlan *plans, const DevOp *ops,
                         const void *tables, bool fp32, void *ws, double err_unit, double *tr, double *kappa, double *err,
                         cudaStream_t st);
// Whether FP_SWEEP_CLUSTER fixes the cluster size of the generic sweep.
bool sweep_cluster_forced();
// Cluster size for a batch whose largest boundary has `bits` bits, and how many
// such clusters can be resident (0 if clusters of that size cannot launch).
int sweep_cluster_size(int bits);
int sweep_max_clusters(int cs, bool fp32);
// FP64 moments per group (deterministic).
cudaError_t launch_moments(const double *tr, const int32_t *group, uint64_t count, int k_max,
                           int n_groups, double *partials, int nblocks, double *out,
                           cudaStream_t st);
int moments_blocks(uint64_t count);
// Bootstrap of F^(k): tr [2 count], group [count] on the device; scratch of
// bootstrap_scratch bytes; out[(g*k_max + k-1)*B + b].  Waits for the group sizes.
size_t bootstrap_scratch(uint64_t count, int n_groups, int k_max, int B);
cudaError_t launch_bootstrap(const double *tr, const int32_t *group, uint64_t count, int n_groups, int k_max, int B,
                             uint64_t seed, void *scratch, double *out, cudaStream_t st);
// Brickwork fast path: maps (from the raw gates; raw == nullptr: they are in place), then either the shared-memory sweep (tile_bits == 0)
// or init + light-cone passes + dot.  `states` holds npairs x 2 x 2^N
// amplitudes (tiled) or npairs x 2^N (shared-memory path, left boundaries).
cudaError_t launch_brick(const BrickDev &d, const BrickPass *hpasses, const BrickDevPlan &dp,
                         const PairInfo *pairs, int npairs, const double2 *raw, void *maps, void *states,
                         bool fp32, double err_scale, double *tr, double *kappa, double *err, cudaStream_t st,
                         int *launches);
size_t brick_smem_bytes(const BrickDev &d, bool fp32, bool *both);
// Tensor-core tile passes (kernels_brick_tc.cu): whether a plan qualifies
// (kTcTile-bit tiles, kMaxWin-bit windows, boundary of more than one tile
// pair), the window-matrix workspace per pair (placed after the boundaries in
// `states`), and the launches of both sides.
bool tc_plan_ok(const BrickDev &d, const BrickPass *hpasses, const RegPass *rps);
size_t tc_wmat_bytes_per_pair(const BrickDev &d, const BrickPass *hpasses);
cudaError_t run_passes_tc(const BrickDev &d, const BrickPass *hpasses, const BrickDevPlan &dp, int npairs,
                          const float2 *maps, float2 *states, float *wm, int *err, cudaStream_t st);
// Spiral sweep (the paper's HEA): maps from merged 1-qubit operators
// (spiral_map_elems(fp32) elements of C per map), then the sweep.  The
// configuration of a state of 2^bits amplitudes: R = 0 applies one map per
// pass (shared memory when it fits, else `scratch`, scratch_elems per pair);
// R = 4 or 5 runs windows of R bits (spiral_windows with `split` cluster bits) over
// shared memory of one CTA (split = 0) or a 2^split-CTA cluster (split <= 2, FP64 <= 4).
constexpr size_t kSpiralSmemMax = 128 * 1024;
struct SpiralConfig {
    int R = 0;
    int split = 0;
    size_t scratch_elems = 0;
};
SpiralConfig spiral_config(int bits, bool fp32, int min_split = 0);   // split >= min_split where it applies
// FP64 clusters of this form that the device holds at a time, and about what a window
// takes them (us): 16-amplitude groups of 3 maps keep an SM quarter busy for 14.8 us per
// warp (an FP64 instruction per 77 cycles), plus the barrier.
int spiral_resident(int bits, const SpiralConfig &cfg);
double spiral_wave_us(int bits, int split);
size_t spiral_map_elems(bool fp32);
cudaError_t launch_spiral(const PairInfo *pairs, int npairs, const SpiralMap *sm, int nmaps, int bits, int first_bit,
                          const SpiralConfig &cfg, const SpiralWin *wins, int nwins, const SpiralCut &cut,
                          const double2 *merged, void *maps, void *scratch, bool fp32, double err_scale, double *tr,
                          double *kappa, double *err, cudaStream_t st);
// Qudit brickwork (kernels_qudit.cu): sampler, maps and sweep of pairs
// pairs[0..npairs) of one depth (BrickDev of the qubit plan with N = 2(l-1)
// q-ary digits); `ws` holds qudit_workspace_per_pair bytes per pair; results
// at slot pairs[i].out of tr/kappa/err.
size_t qudit_workspace_per_pair(int q, const BrickDev &d, bool fp32);
cudaError_t launch_qudit(int q, const BrickDev &d, uint64_t seed, const PairInfo *pairs, int npairs,
                         int self_pair, bool fp32, void *ws, double err_scale, double *tr, double *kappa, double *err,
                         cudaStream_t st);
// Time limit of one bounded device wait (nanoseconds of the global timer):
// fp_set_wait_limit_ns, default 1 s.
uint64_t wait_limit_ns();
// Set the thread-local message returned by fp_last_error().
void set_last_error(const char *msg);
// Internal access for the control-variate driver (cv.cu).
fp_status api_fail(fp_status s, const char *msg);
fp_ensemble_desc ens_desc(const fp_ensemble *E);
cudaStream_t ens_stream(const fp_ensemble *E);
// FP32-policy traces of pairs [first, first+count) into the ensemble's device
// array (*tr_dev, 2*count doubles), device milliseconds into *gpu_ms.
fp_status cv_trace(fp_ensemble *E, uint64_t first, uint64_t count, double **tr_dev, float *gpu_ms);

// BF16 tensor-core GEMM (tc_gemm.cu): C[M x N] = A[M x K] . Bt[N x K]^T (+ bias),
// FP32 accumulation, epilogue mode 0 identity / 1 GELU (pre-activation to Z if
// set) / 2 times GELU'(Z); outputs FP32 row-major (Cf), BF16 row-major (Cb),
// BF16 transposed (Cbt[col * ldct + row]); any subset.  err (device int, may be
// null) is set to 1 if a bounded wait ran out.
struct TcGemm {
    int M, N, K;
    const __nv_bfloat16 *A;
    int lda;
    const __nv_bfloat16 *Bt;
    int ldb;
    const float *bias;
    int mode;
    float *Z;
    int ldz;
    float *Cf;
    int ldcf;
    __nv_bfloat16 *Cb;
    int ldcb;
    __nv_bfloat16 *Cbt;
    int ldct;
    int *err;
    uint64_t wait_ns;   // bounded-wait limit (set at launch from wait_limit_ns())
};
const char *tc_gemm_check(const TcGemm &g);   // nullptr if the arguments are valid
cudaError_t launch_tc_gemm(const TcGemm &g, cudaStream_t st);
size_t tc_gemm_smem_bytes();

}  // namespace fpk
