// Operand staging kernels.
//
// Bound: latency and HBM/L2 (a layer's input is read once and its staged copy written once; a few MB at the usual batch
// sizes).  One launch handles the input and, on calls that bring their filters along, the filters too: the two re-layouts are
// independent, so one of them runs under the other instead of behind it, and a launch less stands in front of the main kernel.
#include <cuda_fp16.h>

#include <algorithm>

#include "stage.h"

namespace boda {
namespace {

constexpr int kThreads = 256;
constexpr int kMaxSmemTaps = 36;             // filter taps staged through shared memory (8 warps x 32 channels x taps floats)

__device__ __forceinline__ float rna(float x)
{
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}

// four consecutive channels of one staged row
template <int MODE>
__device__ __forceinline__ void put4(void* base, size_t row, int Cp, int c, float x0, float x1, float x2, float x3)
{
    if constexpr (MODE == STAGE_F16) {
        const __half2 a = __floats2half2_rn(x0, x1), b = __floats2half2_rn(x2, x3);
        *reinterpret_cast<uint2*>(static_cast<__half*>(base) + row * Cp + c) =
            make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
    } else if constexpr (MODE == STAGE_FP32) {
        *reinterpret_cast<float4*>(static_cast<float*>(base) + row * Cp + c) = make_float4(x0, x1, x2, x3);
    } else {
        float* dst = static_cast<float*>(base) + row * (MODE == STAGE_TF32_SPLIT ? 2 * Cp : Cp) + c;
        const float4 hi = make_float4(rna(x0), rna(x1), rna(x2), rna(x3));
        *reinterpret_cast<float4*>(dst) = hi;
        if constexpr (MODE == STAGE_TF32_SPLIT)
            *reinterpret_cast<float4*>(dst + Cp) = make_float4(rna(x0 - hi.x), rna(x1 - hi.y), rna(x2 - hi.z), rna(x3 - hi.w));
    }
}
template <int MODE>
__device__ __forceinline__ void put1(void* base, size_t row, int Cp, int c, float x)
{
    if constexpr (MODE == STAGE_F16) static_cast<__half*>(base)[row * Cp + c] = __float2half_rn(x);
    else if constexpr (MODE == STAGE_FP32) static_cast<float*>(base)[row * Cp + c] = x;
    else {
        float* dst = static_cast<float*>(base) + row * (MODE == STAGE_TF32_SPLIT ? 2 * Cp : Cp) + c;
        const float hi = rna(x);
        dst[0] = hi;
        if constexpr (MODE == STAGE_TF32_SPLIT) dst[Cp] = rna(x - hi);
    }
}

// Blocks [0, filter_blocks) stage the filters, the rest the input.
// PX: points per input tile (32 channels each).
template <int MODE, int PX>
__global__ void __launch_bounds__(kThreads)
stage_kernel(const StageInput x, const StageFilters w, int filter_blocks, int m_tiles)
{
    extern __shared__ float sm[];
    pdl_launch_dependents();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if ((int)blockIdx.x >= filter_blocks) {
        // ---- input: PX points (numbered through all images) x 32 channels, transposed through shared memory (odd pitch:
        // channel-quad reads hit distinct banks)
        constexpr int PITCH = PX + 1, STEP = kThreads / PX, LOADS = 32 / STEP;
        const int b = (int)blockIdx.x - filter_blocks;
        const int bc = b / m_tiles;
        const int px0 = (b - bc * m_tiles) * PX, c0 = 32 * bc;
        const unsigned M = (unsigned)x.N * (unsigned)x.HW;              // tensors hold at most 2^31 elements
        const int px = tid & (PX - 1), ch = tid / PX;          // channels ch, ch + STEP, ...
        const unsigned m = (unsigned)(px0 + px);
        const bool ok = m < M;
        const unsigned n = ok ? m / (unsigned)x.HW : 0u;
        const float* src = x.in + ((size_t)n * x.C + c0 + ch) * x.HW + (ok ? m - n * (unsigned)x.HW : 0u);
        pdl_wait();
        float v[LOADS];
#pragma unroll
        for (int i = 0; i < LOADS; ++i) v[i] = (ok && c0 + ch + STEP * i < x.C) ? __ldg(src + (size_t)(STEP * i) * x.HW) : 0.f;
#pragma unroll
        for (int i = 0; i < LOADS; ++i) sm[(ch + STEP * i) * PITCH + px] = v[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < PX / 32; ++i) {
            const int p = (tid >> 3) + 32 * i, c = 4 * (tid & 7);
            if ((unsigned)(px0 + p) < M) {
                const float* t = sm + c * PITCH + p;
                put4<MODE>(x.xp, (size_t)px0 + p, x.Cp, c0 + c, t[0], t[PITCH], t[2 * PITCH], t[3 * PITCH]);
            }
        }
        return;
    }
    pdl_wait();
    if (w.RS == 1) {
        // ---- 1x1 filters are [K][C] rows already: a copy with rounding and padding, 512 consecutive channels' worth per warp
        const long long total = (long long)w.K * w.Cp;
        const long long base = ((long long)blockIdx.x * 8 + warp) * 512;
        float v[16];
        const int k0 = (int)(base / w.Cp), r0 = (int)(base - (long long)k0 * w.Cp);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            int k = k0, c = r0 + lane + 32 * i;
            while (c >= w.Cp) { c -= w.Cp; ++k; }
            v[i] = (k < w.K && c < w.C) ? __ldg(w.filt + (size_t)k * w.C + c) : 0.f;
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            int k = k0, c = r0 + lane + 32 * i;
            while (c >= w.Cp) { c -= w.Cp; ++k; }
            if (base + lane + 32 * i < total) put1<MODE>(w.wp, (size_t)k, w.Cp, c, v[i]);
        }
        return;
    }
    // ---- filters: a warp takes 32 channels of one output channel: 32*RS consecutive floats in, RS rows of 32 channels out
    const int cblocks = w.Cp >> 5;
    const long long unit = (long long)blockIdx.x * 8 + warp;
    if (unit >= (long long)w.K * cblocks) return;
    const int k = (int)(unit / cblocks), c0 = 32 * (int)(unit - (long long)k * cblocks);
    const float* src = w.filt + ((size_t)k * w.C + c0) * w.RS;
    const int live = min(32, w.C - c0);                                  // channels that exist (may be 0 or less)
    if (w.RS <= kMaxSmemTaps) {
        float* s = sm + warp * 32 * w.RS;
        const int n = max(live, 0) * w.RS;
        int i = lane;
        for (; i + 96 < 32 * w.RS; i += 128) {
            float v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = i + 32 * u < n ? __ldg(src + i + 32 * u) : 0.f;
#pragma unroll
            for (int u = 0; u < 4; ++u) s[i + 32 * u] = v[u];
        }
        for (; i < 32 * w.RS; i += 32) s[i] = i < n ? __ldg(src + i) : 0.f;
        __syncwarp();
        for (int t = 0; t < w.RS; ++t) put1<MODE>(w.wp, (size_t)t * w.K + k, w.Cp, c0 + lane, s[lane * w.RS + t]);
    } else {
#pragma unroll 4
        for (int t = 0; t < w.RS; ++t)
            put1<MODE>(w.wp, (size_t)t * w.K + k, w.Cp, c0 + lane, lane < live ? __ldg(src + lane * w.RS + t) : 0.f);
    }
}

}  // namespace

int stage_operands(StageMode mode, const StageInput* input, const StageFilters* filters, cudaStream_t stream)
{
    StageInput x = {nullptr, nullptr, 0, 0, 0, 1};
    StageFilters w = {nullptr, nullptr, 0, 0, 0, 1};
    long long fblocks = 0, m_tiles = 1, iblocks = 0;
    size_t smem = 0;
    if (filters) {
        w = *filters;
        if (w.RS == 1) {
            fblocks = ((long long)w.K * w.Cp + 8 * 512 - 1) / (8 * 512);
        } else {
            fblocks = ((long long)w.K * (w.Cp / 32) + 7) / 8;
            if (w.RS <= kMaxSmemTaps) smem = (size_t)8 * 32 * w.RS * sizeof(float);
        }
    }
    // Wide tiles keep more loads in flight per thread and win once they fill the SMs a few times over; below, narrow tiles
    // spread the same loads over more blocks.  Measured, whole layer: 3x3 on 256 channels, 13x13, batch 20 (216 wide tiles)
    // 20.8 us wide, 19.0 narrow; 49x51 on 97 channels (320) 12.7 wide, 13.1 narrow; 39x39 on 333, batch 8 (1140) 15.2 / 18.0.
    // The split staging writes twice as much per load: 41x41 on 32 channels, batch 31 (408) 30.1 wide, 29.4 narrow.
    bool wide = false;
    if (input) {
        x = *input;
        const long long M = (long long)x.N * x.HW;
        wide = (M + 127) / 128 * (x.Cp / 32) >= (mode == STAGE_TF32_SPLIT ? 148 * 8 : 148 * 2);
        const int px = wide ? 128 : 32;
        m_tiles = (M + px - 1) / px;
        iblocks = m_tiles * (x.Cp / 32);
        smem = std::max(smem, (size_t)32 * (px + 1) * sizeof(float));
    }
    if (fblocks + iblocks > 0x7fffffffLL || m_tiles > 0x7fffffffLL) return BODA_ERR_TOO_LARGE;
    const dim3 grid((unsigned)(fblocks + iblocks)), block(kThreads);
    auto run = [&](auto narrow_kernel, auto wide_kernel) {
        return launch_kernel(wide ? wide_kernel : narrow_kernel, grid, block, smem, stream, 1, x, w, (int)fblocks, (int)m_tiles);
    };
    cudaError_t e;
    switch (mode) {
        case STAGE_TF32: e = run(stage_kernel<STAGE_TF32, 32>, stage_kernel<STAGE_TF32, 128>); break;
        case STAGE_TF32_SPLIT: e = run(stage_kernel<STAGE_TF32_SPLIT, 32>, stage_kernel<STAGE_TF32_SPLIT, 128>); break;
        case STAGE_F16: e = run(stage_kernel<STAGE_F16, 32>, stage_kernel<STAGE_F16, 128>); break;
        default: e = run(stage_kernel<STAGE_FP32, 32>, stage_kernel<STAGE_FP32, 128>); break;
    }
    if (e != cudaSuccess) return record_cuda_error(e, "stage_kernel");
    count_launch();
    return BODA_OK;
}

}  // namespace boda
