// fp32 passes with the block kernels in registers (harp_regs.cu), as harp_f32.cu plans and launches them.
#pragma once

#include "harp_internal.h"

struct RegPass {
    int32_t shape;             // number of its kernel, 0: none
    int32_t n_lo, n_cg;        // groups of neighbouring coordinates below the stride; column groups
    int32_t linear;            // whole rows as one run of memory
    int64_t S, d;              // stride of the first stage
    int64_t off[11];           // the stages' offsets in the plan's block array
};

bool harp_regs_pass(const StageTable &st, int64_t d, int t0, int t1, bool col, RegPass &P);
// n vectors: rows ld apart (blocks: the element-major copy), or columns of a matrix whose rows are ld apart (block after block).  signs: of the pass's first stage (forward: operands, transpose: results)
cudaError_t harp_regs_launch(void *encode, const RegPass &P, int sms, float *x, int64_t n, int64_t ld, const float *blocks, const int8_t *signs, int transpose,
                             int32_t *err, cudaStream_t stream);

// one stage of radix 17 to 48 over rows (harp_big.cu; blocks: block after block)
constexpr int kBigShape = 1000;        // shape = kBigShape + radix
bool harp_big_pass(const StageTable &st, int64_t d, int t, RegPass &P);
cudaError_t harp_big_launch(void *encode, const RegPass &P, int sms, float *x, int64_t n, int64_t ld, const float *blocks, int transpose, int32_t *err,
                            cudaStream_t stream);
