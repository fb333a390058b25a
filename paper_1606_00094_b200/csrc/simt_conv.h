// FP32 convolution over a staged NHWC copy of the input (CUDA cores, TMA-fed): host-side interface.
#pragma once

#include "boda_internal.h"

namespace boda {

struct SimtPlan;

// bn: output channels per tile, 128, 96, 64, 48 or 32.  simt_legal: false for windows or pads the im2col loads do not take.
bool simt_legal(const ConvDims& d);
double simt_cost(const ConvDims& d, int bn);                 // estimated SM clocks of one call, staging included
size_t simt_workspace_bytes(const ConvDims& d, int bn);
int simt_plan_create(const ConvDims& d, int bn, int* d_status, SimtPlan** out);
void simt_plan_destroy(SimtPlan* p);
void simt_plan_describe(const SimtPlan* p, char* buf, size_t n);
int simt_plan_kernels(const SimtPlan* p);                    // launches per call
int simt_launch(SimtPlan* p, const float* in, const float* filt, const float* bias, float* out, void* workspace, cudaStream_t stream,
                cudaEvent_t after_staging);

}  // namespace boda
