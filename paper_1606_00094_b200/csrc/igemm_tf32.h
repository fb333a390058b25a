// Tensor-core (tcgen05, TF32) implicit-GEMM variants K1CONV and TCONV: host-side interface.
#pragma once

#include "boda_internal.h"

namespace boda {

struct IgemmPlan;

bool igemm_variant_legal(const ConvDims& d, int variant);
// Rule used by automatic selection: is the tensor-core path expected to beat DIRECT for this shape?
bool igemm_variant_profitable(const ConvDims& d);
// What the tensor-core kernels cost in the TF32 mode as the line between FP32 and TF32 layers counts (estimated SM clocks, staging of the input
// included), and what the kernel meant reads: a staged copy, NCHW gathered by warps, or NCHW by TMA.  Allocates nothing.
enum IgemmKind { IGEMM_STAGES = 0, IGEMM_GATHERS = 1, IGEMM_READS_NCHW = 2 };
double igemm_rule_cost(const ConvDims& d, int variant, size_t max_ws, IgemmKind* kind);
int igemm_num_tiles();
int igemm_num_split_candidates();
int igemm_split_candidate(int i);

// s2d: -1 automatic, 0 never, 1 force the space-to-depth view of a strided tconv layer.
// mode: 0 TF32; 1 error-compensated TF32 (three tensor-core products per FP32 product); 2 fp16 operands (fp32
// accumulate).  Mode 1: split operands or the im2col kernel, mode 2: im2col, pair and slab kernels; NCHW in and out.
// max_ws: 0, or the largest workspace (staged input) the caller accepts; BODA_ERR_NOMEM if no tile fits it.  use: in a chain, kernels that read NCHW only
// are not chosen by rule where they would part the layer from its neighbours' staged layouts.
int igemm_plan_create(const ConvDims& d, int variant, int tile_id, int split_k, int s2d, int* d_status, IgemmPlan** out,
                      int mode = 0, size_t max_ws = 0, PlanUse use = PLAN_ALONE);
bool igemm_s2d_applicable(const ConvDims& d);
void igemm_plan_destroy(IgemmPlan* p);
int igemm_plan_tile(const IgemmPlan* p);
// split operands in the place of FP32 arithmetic: short reductions, whose FP32 sums are off by least, are added chunk by chunk
void igemm_plan_fp32_sums(IgemmPlan* p);
bool igemm_plan_writes_packed(const IgemmPlan* p);       // can the plan write a consumer's staged layout?
int igemm_plan_kernels_per_call(const IgemmPlan* p);     // 1, or 2 where an input staging kernel runs first
int igemm_plan_splits(const IgemmPlan* p);
// a tile whose accumulators would take more MMA steps than the error bars allow: run when forced, never picked
bool igemm_plan_sums_too_long(const IgemmPlan* p);
size_t igemm_plan_workspace_bytes(const IgemmPlan* p);
void igemm_plan_describe(const IgemmPlan* p, char* buf, size_t n);
int igemm_bind_filters(IgemmPlan* p, const float* filt, cudaStream_t stream);
void igemm_unbind_filters(IgemmPlan* p);
// after_staging (may be null): event recorded on the stream between the operand-staging kernels and the main kernel
int igemm_launch(IgemmPlan* p, const float* in, const float* filt, const float* bias, float* out, void* workspace,
                 cudaStream_t stream, cudaEvent_t after_staging = nullptr);

// The split-operand tiles (error-compensated mode, FP32 accuracy): may they run the shape, the estimated SM clocks of one call with its
// best split, staging of both operands included (`clocks`: by a second model), and the workspace they need.
bool igemm_split_legal(const ConvDims& d);
double igemm_split_cost(const ConvDims& d, int tile, double* clocks);
size_t igemm_split_workspace(const ConvDims& d);
// the most that automatic selection and the tuner let these tiles take where the caller sets no limit
size_t igemm_split_workspace_limit(const ConvDims& d);
bool igemm_tile_is_split(int tile);
bool igemm_tile_is_slab(int tile);
// Does a kernel other than the slab kernel (mode 0 or 2) run the layer under these options?  Slabs, which take no workspace, are no reason to run one that a limit
// on it rules out.
bool igemm_runs_without_slabs(const ConvDims& d, int variant, int split_k, int s2d, int mode, size_t max_ws);

// Activation layouts for chained layers.  igemm_plan_input_geometry: the staged input layout this plan reads,
// rows [(n*Hp + y)*Wp + x][Cp] (false if the plan cannot take a staged input).  igemm_plan_set_io: in_packed =
// the `in` pointer of igemm_launch already is that layout (no staging kernel, no workspace); out_packed = write
// the output as rows [(n*oHp + p)*oWp + q][oCp] rounded to TF32 instead of NCHW.
bool igemm_plan_input_geometry(const IgemmPlan* p, int* Hp, int* Wp, int* Cp);
int igemm_plan_set_io(IgemmPlan* p, int in_packed, int out_packed, int oHp, int oWp, int oCp);

// Fused ReLU -> 3x3 / stride-2 max-pooling in the epilogue (halo tiles with 2 or 4 accumulators, no split): the plan
// then writes the POOLED tensor (out_packed geometry and NCHW extents refer to it).  set_pool(p, 0, 0) undoes it.
// Call set_pool before set_io.
bool igemm_plan_can_fuse_pool(const IgemmPlan* p, int ksz, int stride);
int igemm_plan_set_pool(IgemmPlan* p, int ksz, int stride);
void igemm_plan_pooled_dims(const IgemmPlan* p, int* P, int* Q);

// Scratch-in-a-caller-region form (allocates nothing): bytes needed at least, and the run itself.
size_t igemm_region_min_bytes(const ConvDims& d);
int igemm_run_in_region(const ConvDims& d, int variant, const float* in, const float* filt, const float* bias,
                        float* out, void* region, size_t region_bytes, cudaStream_t stream);

}  // namespace boda
