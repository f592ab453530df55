// Internal declarations shared by the translation units of libharp.so.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <vector>

#include "harp.h"

#define HARP_MAX_STAGES 24

// Stage geometry handed to kernels by value.
struct StageTable {
    int32_t m;
    int32_t b[HARP_MAX_STAGES];       // radix b_t
    int32_t s[HARP_MAX_STAGES];       // stride s_t = prod_{j<t} b_j
    int64_t off[HARP_MAX_STAGES];     // offset (in floats) of stage t in the block array
};

struct FastPlan;   // tensor-core path data, whole rows per CTA (harp_fast.cu)
struct SplitPlan;  // tensor-core path data, two passes over column groups (harp_split.cu)
struct TmPlan;    // tensor-memory path data: tcgen05.mma, rows as the M dimension (harp_tm.cu)
struct F32Plan;    // CUDA-core passes over column groups for fp32 rows and matrices (harp_f32.cu)
struct ColPlan;    // tensor-core path data for applying the plan down the columns of a matrix (harp_col.cu)

struct harp_plan {
    int64_t d = 0;
    int device = 0;
    StageTable st{};
    int64_t n_params = 0;
    float *d_blocks = nullptr;        // [sum_t d*b_t] fp32, stage after stage
    float *d_blocks_em = nullptr;     // the same stages element-major: entry k of block c of stage t at off[t] + k*D_t + c
    // the same map with runs of small-radix stages fused into dense blocks of size <= 4 (fewer
    // stages for the CUDA-core kernel); fused.m == 0 if nothing could be fused
    StageTable fused{};
    float *d_fused_blocks = nullptr;
    // block kernels of the stage table the block-owner kernels use (fused if present, else st),
    // element-major: entry k = i*b + j of block c of stage t at off[t] + k * (d / b_t) + c, so that
    // neighbouring threads (neighbouring blocks) read neighbouring words
    float *d_bo_blocks = nullptr;
    int32_t *d_perm = nullptr;        // nullptr = identity
    int8_t *d_signs = nullptr;        // nullptr = all +1
    // host copies (used to derive kernel-specific layouts)
    std::vector<int32_t> h_perm;
    std::vector<int8_t> h_signs;
    std::vector<float> h_blocks;
    FastPlan *fast = nullptr;
    SplitPlan *split = nullptr;
    ColPlan *col = nullptr;
    TmPlan *tm = nullptr;
    F32Plan *f32 = nullptr;
    // test-only switches, read from the environment once, when the plan is built (HARP_NO_ROWVEC=1: the
    // CUDA-core kernels keep their tile row-major; HARP_NO_TENSOR_MAPS=1: as on a driver that cannot encode tensor maps;
    // HARP_F32_PASSES=1: fp32 rows take the passes over column groups whatever the batch)
    bool opt_no_rowvec = false, opt_no_maps = false, opt_f32_passes = false;
    // most bytes of states that a gradient asks for (HARP_GRAD_SCRATCH_MB, read then too)
    int64_t opt_grad_scratch = INT64_MAX;
    // staging owned by harp_apply_host
    static constexpr int kStages = 4;
    void *stage_buf[kStages] = {nullptr, nullptr, nullptr, nullptr};
    int64_t stage_bytes = 0;
    cudaStream_t stage_stream[kStages] = {nullptr, nullptr, nullptr, nullptr};
};

extern std::atomic<int64_t> g_harp_launches;

// generic CUDA-core path (harp_generic.cu)
harp_status_t harp_generic_build(harp_plan *plan);   // fused stage table for the block-owner kernel
int harp_generic_max_radix(const harp_plan *plan);   // of the stage table its kernels run
// Estimated microseconds of an fp32 batch on these kernels (harp_f32_preferred: on the passes over column groups), for the choice between
// them: waves of CTAs times a CTA's time.  The constants are fitted to 1235 batches measured on both (d = 72 .. 32768, radices 2 .. 43,
// 1 .. 4096 rows, identity and random permutation): standard deviation 12 % for the passes of harp_f32.cu, 4 to 8 % here up to radix 8, 23 % above it.
// (the passes of harp_regs.cu and harp_big.cu: a launch and a rate, measured at 1 to 4096 rows)
double harp_generic_estimate(const harp_plan *plan, int64_t n_rows, int sms);
harp_status_t harp_generic_supported(const harp_plan *plan, harp_dtype_t dtype);
harp_status_t harp_generic_apply(const harp_plan *plan, void *x, int64_t n_rows, harp_dtype_t dtype,
                                 int transpose, cudaStream_t stream);

// tensor-core path (harp_fast.cu)
harp_status_t harp_fast_build(harp_plan *plan);     // HARP_OK or HARP_ERR_UNSUPPORTED (plan->fast stays null)
void harp_fast_destroy(harp_plan *plan);
int32_t harp_fast_error_word(const harp_plan *plan);
bool harp_fast_yields(const harp_plan *plan, int64_t n_rows);   // the two-pass path is faster for this batch
harp_status_t harp_fast_apply(const harp_plan *plan, void *x, int64_t n_rows, harp_dtype_t dtype,
                              int transpose, cudaStream_t stream);

// tensor-core path for wide rows (harp_split.cu)
harp_status_t harp_split_build(harp_plan *plan);
void harp_split_destroy(harp_plan *plan);
int32_t harp_split_error_word(const harp_plan *plan);
bool harp_split_piped(const harp_plan *plan);       // both passes have kernels fed by the copy engine
harp_status_t harp_split_apply(const harp_plan *plan, void *x, int64_t n_rows, harp_dtype_t dtype,
                               int transpose, cudaStream_t stream);

// tensor-memory path (harp_tm.cu)
harp_status_t harp_tm_build(harp_plan *plan);
void harp_tm_destroy(harp_plan *plan);
harp_status_t harp_tm_apply(const harp_plan *plan, void *x, int64_t n_rows, harp_dtype_t dtype,
                            int transpose, cudaStream_t stream);
// cuTensorMapEncodeTiled of the driver (null if it has none, or for a plan built without: HARP_NO_TENSOR_MAPS)
void *harp_tensor_map_encoder(const harp_plan *plan);
int32_t harp_tm_error_word(const harp_plan *plan);
// the stages below stride 256 alone (lower pass of the two-pass paths); 0 stages = not available
int harp_tm_slab_stages(const harp_plan *plan);
harp_status_t harp_tm_slab_apply(const harp_plan *plan, void *x, int64_t n_rows, harp_dtype_t dtype,
                                 int transpose, cudaStream_t stream);

// column-side apply for two-sided processing (harp_col.cu): plan applied down the columns of a
// dim(plan) x n_cols row-major matrix with leading dimension ld
harp_status_t harp_col_build(harp_plan *plan);
void harp_col_destroy(harp_plan *plan);
int32_t harp_col_error_word(const harp_plan *plan);
harp_status_t harp_col_apply(const harp_plan *plan, void *W, int64_t n_cols, int64_t ld, harp_dtype_t dtype,
                             cudaStream_t stream);

// fp32 passes over column groups (harp_f32.cu): rows, and down the columns of a row-major matrix
harp_status_t harp_f32_build(harp_plan *plan);
void harp_f32_destroy(harp_plan *plan);
int32_t harp_f32_error_word(const harp_plan *plan);
// source of every coordinate under the plan's permutation, its sign in the top bit (device; null: none, or a plan without fp32 passes)
const int32_t *harp_f32_source_table(const harp_plan *plan);
bool harp_f32_preferred(const harp_plan *plan, int64_t n_rows);      // faster than the whole-row kernels, by the estimates
harp_status_t harp_f32_apply(const harp_plan *plan, void *x, int64_t n_rows, harp_dtype_t dtype, int transpose,
                             cudaStream_t stream);
harp_status_t harp_f32_col_apply(const harp_plan *plan, void *W, int64_t n_cols, int64_t ld, harp_dtype_t dtype,
                                 cudaStream_t stream);

// out-of-place matrix transpose, rows x cols -> cols x rows (harp_two_sided.cu)
harp_status_t harp_transpose_matrix(const void *src, void *dst, int64_t rows, int64_t cols,
                                    harp_dtype_t dtype, cudaStream_t stream);

static inline size_t harp_dtype_size(harp_dtype_t t) { return t == HARP_F32 ? 4 : 2; }
