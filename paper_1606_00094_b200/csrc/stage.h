// Operand staging: the input and filter re-layouts ("input transformation", Section 5 of the paper) that the kernels
// reading NHWC rows need, both in one launch.
#pragma once

#include "boda_internal.h"

namespace boda {

// What the staged operands hold.  TF32: values rounded to TF32 (nearest, ties away), so that the tensor core's truncation of
// the low mantissa bits is exact.  TF32_SPLIT: rows of 2*Cp values, the rounded value hi at channel c and the rounded
// remainder lo = rna(x - hi) at channel Cp + c (x = hi + lo up to 2^-22 relative).  F16: nearest fp16.  FP32: as they are.
// BF16X3: rows of 3*Cp bf16 values, x = h + m + l exactly: x rounded to bf16 (nearest even) at channel c, the rest rounded at Cp + c, what is
// left then at 2*Cp + c (m and l of an infinity or NaN are zero).
enum StageMode { STAGE_TF32 = 0, STAGE_TF32_SPLIT = 1, STAGE_F16 = 2, STAGE_FP32 = 3, STAGE_BF16X3 = 4 };

struct StageInput { const float* in; void* xp; int N, C, Cp, HW; };           // NCHW -> rows [(n*HW + hw)][Cp], channels past C zero
struct StageFilters { const float* filt; void* wp; int K, C, Cp, RS; };       // KCRS -> [RS][K][Cp], channels past C zero

// Either part may be null.  Cp is a multiple of 32.  Counts one launch.
int stage_operands(StageMode mode, const StageInput* input, const StageFilters* filters, cudaStream_t stream);

}  // namespace boda
