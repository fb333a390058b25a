// Operand staging: the input and filter re-layouts ("input transformation", Section 5 of the paper) that the kernels
// reading NHWC rows need, both in one launch.
#pragma once

#include "boda_internal.h"

namespace boda {

// What the staged operands hold.  TF32: values rounded to TF32 (nearest, ties away), so that the tensor core's truncation of
// the low mantissa bits is exact.  TF32_SPLIT: rows of 2*Cp values, the rounded value hi at channel c and the rounded
// remainder lo = rna(x - hi) at channel Cp + c (x = hi + lo up to 2^-22 relative).  F16: nearest fp16.  FP32: as they are.
// BF16X3: rows of 3*Cp bf16 values, x = h + m + l exactly: x rounded to bf16 (nearest even) at channel c, the rest rounded at Cp + c, what is
// left then at 2*Cp + c (m and l of an infinity or NaN are zero).  The rest is multiplied by kPartScale before each rounding, x = h + m / 2^7 +
// l / 2^14, which makes the parts about as large as x: operands down to 2^-124 keep all their bits (the smallest bf16 value is 2^-133) and no
// operand loses more than 2^-148.  (Unscaled, l begins to go below 2^-110: operands around 2^-120 were off by 7e-5 of themselves.)  Not more
// than 2^7: |h*m + m*h| stays within |x*w|, so that these sums overflow no earlier than those of h*h.
constexpr float kPartScale = 128.f;
enum StageMode { STAGE_TF32 = 0, STAGE_TF32_SPLIT = 1, STAGE_F16 = 2, STAGE_FP32 = 3, STAGE_BF16X3 = 4 };

struct StageInput { const float* in; void* xp; int N, C, Cp, HW; };           // NCHW -> rows [(n*HW + hw)][Cp], channels past C zero
struct StageFilters { const float* filt; void* wp; int K, C, Cp, RS; };       // KCRS -> [RS][K][Cp], channels past C zero

// Either part may be null.  Cp is a multiple of 32.  Counts one launch.
int stage_operands(StageMode mode, const StageInput* input, const StageFilters* filters, cudaStream_t stream);

}  // namespace boda
