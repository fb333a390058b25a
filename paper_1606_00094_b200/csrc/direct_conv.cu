// DIRECT variant: FP32 CUDA-core convolution, the general fallback (the paper's `conv`, Section 5:
// SGEMM blocking with im2col folded into the shared-memory load) and the small-input-channel path.
//
// Blocking follows the paper's SGEMM template (Section 4, Listing 1 and the parameter list after
// it): each thread owns a register tile of Mt x Nt outputs (here TM pixels x TN output channels),
// a thread block of WM x WN warps (8 x 4 lanes each) owns (8*WM*TM) x (4*WN*TN) outputs, the reduction is
// walked in chunks of Kb = BK, operands of a chunk are staged in shared memory and the inner loop
// is fully unrolled.  The gather that im2col would do is a table lookup: entry j of the table
// gives, for reduction index j = (c, r, s), the element offset inside an image and the tap, so the
// load needs no division.  Bias and ReLU are applied in registers before the store.
#include <algorithm>
#include <cmath>

#include "boda_internal.h"
#include "igemm_tf32.h"
#include "simt_conv.h"

namespace boda {
namespace {

// ---- GEMM-blocked form.  Bound: the FP32 pipe (128 multiply-adds per clock and SM).  What keeps it busy:
//  * multiply-adds in pairs (__ffma2_rn, each half rounds like fmaf) along the REDUCTION: the two halves of an accumulator
//    are the sums over the even and the odd reduction indices and are added once at the end.  Input pixels and weights both
//    sit in shared memory as such pairs, so nothing is broadcast or moved between registers;
//  * operands of a chunk arrive by asynchronous copies, kStages - 1 chunks ahead, straight into shared memory (no
//    registers held, zero fill for the padding and the ragged ends);
//  * the reduction is split over the CTAs of a cluster (grid.z) where the output tiles alone would leave SMs idle or the
//    last wave thin; the partial tiles are summed in rank order through distributed shared memory, so every run gives the
//    same bits.
//  * the next kernel is let in when the reduction is through, not at once: blocks that wait for this kernel take the places that its own
//    leave free, wherever those are, and sit there unevenly when their turn comes.  Call after call, 5x5 on 3 channels, 15 filters,
//    55x57, batch 4: 9.4 / 5.2 us; 3x3 on 49 channels, 114 filters, 10x10, batch 4: 11.1 / 6.0; without programmatic launch 8.2 both.
// Measured (before / now): 5x5 on 23 channels, 87 filters, 11x11, batch 3 (0.04 GFLOP) 33 / 6.4 us; 3x3 on 200 channels, 48
// filters, 14x14, batch 8 (0.27 GFLOP) 54 / 22 us.  Large layers run over a staged input instead (simt_conv.cu).
constexpr int kStages = 4;
constexpr int kMaxSplit = 8;
// windows whose bounds tests fit a 32-bit mask per pixel: bit tap + 2 set = inside the image, so that (mask >> tap) & 4 is the
// byte count of the copy.  Entries past the end of the reduction carry tap 29, whose bit is never set.
constexpr int kMaskTaps = 29;

template <int WM, int WN, int TM, int TN, int BK>
struct GemmCfg {
    static constexpr int THREADS = 32 * WM * WN;
    static constexpr int BM = 8 * WM * TM, BN = 4 * WN * TN;
    static constexpr int APITCH = 2 * BM, BPITCH = 2 * BN + 4;     // floats of one row of index pairs; +4: the copies hit distinct banks
    static constexpr int BMP = BM + 4;                 // pitch of a finished channel row
    static constexpr int STAGE_FLOATS = BK / 2 * (APITCH + BPITCH);
    static constexpr int SMEM_FLOATS = kStages * STAGE_FLOATS > BN * BMP ? kStages * STAGE_FLOATS : BN * BMP;
    static constexpr int SMEM_BYTES = SMEM_FLOATS * 4;
    // 64 accumulator registers fit 128 registers a thread, 96 fit 168
    static constexpr int BLOCKS_PER_SM = (TM * TN <= 32 ? 512 : TM * TN <= 48 ? 320 : 256) / THREADS;
};

// 4 or 8 bytes, or zeros where `bytes` is 0 (the source is then not read)
__device__ __forceinline__ void copy4_async(uint32_t dst, const float* src, uint32_t bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" :: "r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void copy8_async(uint32_t dst, const float* src, uint32_t bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" :: "r"(dst), "l"(src), "r"(bytes) : "memory");
}
template <int WM, int WN, int TM, int TN, int BK, bool MASKED>
__global__ void __launch_bounds__(GemmCfg<WM, WN, TM, TN, BK>::THREADS, GemmCfg<WM, WN, TM, TN, BK>::BLOCKS_PER_SM)
direct_conv_kernel(const ConvDims d, const float* __restrict__ in, const float* __restrict__ filt,
                   const float* __restrict__ bias, float* __restrict__ out,
                   const DirectTapEntry* __restrict__ tab, int chunks_total, int chunks_per_split)
{
    using G = GemmCfg<WM, WN, TM, TN, BK>;
    constexpr int BM = G::BM, BN = G::BN, BMP = G::BMP, NT = G::THREADS;
    static_assert(NT % BM == 0 && NT % BK == 0 && BN % (NT / BK) == 0 && BK % (NT / BM) == 0, "the copies are dealt without a remainder");
    static_assert(TM % 2 == 0 && TN % 2 == 0 && BK % 2 == 0, "16-byte loads hold two pixels or two channels of an index pair");
    constexpr int A_STEP = NT / BM, A_PER = BK / A_STEP;          // a thread copies one pixel's indices a_kk0, a_kk0 + A_STEP, ...
    constexpr int B_STEP = NT / BK, B_PER = BN / B_STEP;          // and one index of channels b_n0, b_n0 + B_STEP, ...
    constexpr int B2_STEP = 2 * B_STEP, B2_PER = (BN + B2_STEP - 1) / B2_STEP;      // or one index pair of half as many
    extern __shared__ __align__(16) float sm_gemm[];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // lane bits 1, 3, 4 -> pixel group, bits 0, 2 -> channel group: lanes i and i^1 read the same pixels and lanes i and i^2 the
    // same weights, which lets a 16-byte shared-memory load serve two quarter warps at once
    const int lane_m = ((lane >> 1) & 1) | ((lane >> 2) & 6), lane_n = (lane & 1) | ((lane >> 1) & 2);
    const int wm = warp % WM, wn = warp / WM;
    const int m0 = blockIdx.x * BM;
    const int k0 = blockIdx.y * BN;
    const int PQ = d.P * d.Q;
    const int HW = d.H * d.W;
    const int t_begin = (int)blockIdx.z * chunks_per_split;
    const int chunks = min(chunks_total - t_begin, chunks_per_split);

    // ---- per-thread constants of the A (input) gather: this thread always copies pixel ml
    const int ml = tid % BM;
    const int a_kk0 = tid / BM;
    int a_y0 = 0, a_x0 = 0, img = 0, pq = 0;
    const float* a_ptr = in;
    const bool m_ok = m0 + ml < d.M;
    uint32_t taps_in = 0;                      // see kMaskTaps
    {
        const int m = m_ok ? m0 + ml : 0;
        img = m / PQ;
        pq = m - img * PQ;
        const int p = pq / d.Q;
        const int q = pq - p * d.Q;
        a_y0 = m_ok ? p * d.stride - d.pad : -0x100000;            // pixels past the end fail every bounds test
        a_x0 = q * d.stride - d.pad;
        a_ptr = in + (long long)img * d.C * HW + (long long)(p * d.stride - d.pad) * d.W + a_x0;
        if constexpr (MASKED) {
            uint32_t bit = 4;
            for (int r = 0; r < d.R; ++r)
                for (int sx = 0; sx < d.S; ++sx, bit <<= 1)
                    if ((unsigned)(a_y0 + r) < (unsigned)d.H && (unsigned)(a_x0 + sx) < (unsigned)d.W) taps_in |= bit;
        }
    }
    // ---- per-thread constants of the B (filter) copy: index pairs as 8-byte copies where every filter row allows it
    const bool pairs = (d.Kred & 1) == 0 && (reinterpret_cast<uintptr_t>(filt) & 7) == 0;
    const int b_kk = pairs ? 2 * (tid % (BK / 2)) : tid % BK;
    const int b_n0 = pairs ? tid / (BK / 2) : tid / BK;
    const float* b_ptr = filt + (size_t)(k0 + b_n0) * d.Kred + t_begin * BK + b_kk;
    const int b_step = pairs ? B2_STEP : B_STEP;
    const size_t b_pitch = (size_t)b_step * d.Kred;
    const int b_rows = (d.K - k0 - b_n0 + b_step - 1) / b_step;                       // of this thread's channels, those that exist
    const uint32_t sm_base = (uint32_t)__cvta_generic_to_shared(sm_gemm);
    const uint32_t a_dst = sm_base + 4u * (uint32_t)((a_kk0 >> 1) * G::APITCH + 2 * ml + (a_kk0 & 1));
    const uint32_t b_dst = sm_base + 4u * (uint32_t)(BK / 2 * G::APITCH + (b_kk >> 1) * G::BPITCH + 2 * b_n0 + (b_kk & 1));
    // the table entries of the next chunk are fetched one chunk early: their latency is off the path of the copies
    DirectTapEntry e[A_PER];
    const DirectTapEntry* my_tab = tab + a_kk0 + t_begin * BK;
#pragma unroll
    for (int i = 0; i < A_PER; ++i) e[i] = my_tab[i * A_STEP];

    auto issue = [&](int t, int buf) {
        const uint32_t off = 4u * (uint32_t)(buf * G::STAGE_FLOATS);
#pragma unroll
        for (int i = 0; i < A_PER; ++i) {
            uint32_t bytes;
            if constexpr (MASKED) {
                bytes = (taps_in >> e[i].rs) & 4u;
            } else {
                const int y = a_y0 + (e[i].rs >> 16);
                const int x = a_x0 + (e[i].rs & 0xffff);
                bytes = ((unsigned)y < (unsigned)d.H && (unsigned)x < (unsigned)d.W) ? 4u : 0u;
            }
            // index a_kk0 + i*A_STEP: a_kk0 < A_STEP, which is 1 or even, so its pair and half are known up to a_kk0's
            const int kk = i * A_STEP;
            copy4_async(a_dst + off + 4u * (uint32_t)((kk >> 1) * G::APITCH + (kk & 1)), a_ptr + e[i].offset, bytes);
        }
        // (the last chunk fetches its own entries once more)
        const DirectTapEntry* nt = my_tab + min(t + 1, chunks - 1) * BK;
#pragma unroll
        for (int i = 0; i < A_PER; ++i) e[i] = nt[i * A_STEP];
        const float* bp = b_ptr;
        b_ptr += BK;
        const bool j_ok = (t_begin + t) * BK + b_kk < d.Kred;       // an even Kred ends on a pair
        if (pairs) {
#pragma unroll
            for (int i = 0; i < B2_PER; ++i) {
                if (B2_PER * B2_STEP > BN && b_n0 + i * B2_STEP >= BN) break;
                copy8_async(b_dst + off + 8u * (uint32_t)(i * B2_STEP), bp, j_ok && i < b_rows ? 8u : 0u);
                bp += b_pitch;
            }
        } else {
#pragma unroll
            for (int i = 0; i < B_PER; ++i) {
                copy4_async(b_dst + off + 8u * (uint32_t)(i * B_STEP), bp, j_ok && i < b_rows ? 4u : 0u);
                bp += b_pitch;
            }
        }
    };

    // accumulators: (sum over even indices, sum over odd indices) of each pixel and channel
    float2 acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = make_float2(0.f, 0.f);

    // pixel 2g + i of this thread is wm*8*TM + 16g + 2*lane_m + i, channel 2h + i is wn*4*TN + 8h + 2*lane_n + i: every warp
    // load is one contiguous run of shared memory
    const int a_rd = wm * 8 * TM + 2 * lane_m, b_rd = wn * 4 * TN + 2 * lane_n;

    pdl_wait();
#pragma unroll
    for (int s = 0; s < kStages - 1; ++s) {
        if (s < chunks) issue(s, s);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    int buf = 0;
    for (int t = 0; t < chunks; ++t) {
        asm volatile("cp.async.wait_group %0;" :: "n"(kStages - 2) : "memory");
        __syncthreads();
        const float* As = sm_gemm + buf * G::STAGE_FLOATS;
        const float* Bs = As + BK / 2 * G::APITCH;
        // operands of the next index pair are loaded while this one's multiply-adds run
        float2 a[2][TM], b[2][TN];
        auto fetch = [&](int k2, float2 (&ao)[TM], float2 (&bo)[TN]) {
#pragma unroll
            for (int g = 0; g < TM / 2; ++g) {
                const float4 v = *reinterpret_cast<const float4*>(As + k2 * G::APITCH + 2 * (a_rd + 16 * g));
                ao[2 * g] = make_float2(v.x, v.y); ao[2 * g + 1] = make_float2(v.z, v.w);
            }
#pragma unroll
            for (int h = 0; h < TN / 2; ++h) {
                const float4 v = *reinterpret_cast<const float4*>(Bs + k2 * G::BPITCH + 2 * (b_rd + 8 * h));
                bo[2 * h] = make_float2(v.x, v.y); bo[2 * h + 1] = make_float2(v.z, v.w);
            }
        };
        fetch(0, a[0], b[0]);
#pragma unroll
        for (int k2 = 0; k2 < BK / 2; ++k2) {
            if (k2 + 1 < BK / 2) fetch(k2 + 1, a[(k2 + 1) & 1], b[(k2 + 1) & 1]);
            // the copies of a later chunk go out under the first multiply-adds
            if (k2 == 0) {
                if (t + kStages - 1 < chunks) issue(t + kStages - 1, (buf + kStages - 1) % kStages);
                asm volatile("cp.async.commit_group;" ::: "memory");
            }
#pragma unroll
            for (int j = 0; j < TN; ++j)
#pragma unroll
                for (int i = 0; i < TM; ++i) acc[i][j] = __ffma2_rn(a[k2 & 1][i], b[k2 & 1][j], acc[i][j]);
        }
        buf = buf + 1 == kStages ? 0 : buf + 1;
    }

    // ---- epilogue: the tile goes through shared memory as [channel][pixel], so that the NCHW stores (and a split's remote
    // reads) are whole 128-byte runs whatever the register blocking
    pdl_launch_dependents();
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
#pragma unroll
    for (int j = 0; j < TN; ++j)
#pragma unroll
        for (int g = 0; g < TM / 2; ++g)
            *reinterpret_cast<float2*>(sm_gemm + (b_rd + 8 * (j >> 1) + (j & 1)) * BMP + a_rd + 16 * g) =
                make_float2(acc[2 * g][j].x + acc[2 * g][j].y, acc[2 * g + 1][j].x + acc[2 * g + 1][j].y);
    const int splits = (int)gridDim.z;
    int n_begin = 0, n_end = BN;
    uint32_t peer[kMaxSplit];
    if (splits > 1) {
        const int share = (BN + splits - 1) / splits;
        n_begin = (int)blockIdx.z * share;
        n_end = min(BN, n_begin + share);
#pragma unroll
        for (int r = 0; r < kMaxSplit; ++r)
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(peer[r]) : "r"(sm_base), "r"(r < splits ? r : 0));
        asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    } else {
        __syncthreads();
    }
    n_end = min(n_end, d.K - k0);
    float* o = out + ((size_t)img * d.K + k0) * PQ + pq;
    auto finish = [&](int nl, float v) {
        v += bias ? __ldg(bias + k0 + nl) : 0.f;
        if (d.relu) v = fmaxf(v, 0.f);
        o[(size_t)nl * PQ] = v;
    };
    if (m_ok) {
        if (splits == 1) {
#pragma unroll 4
            for (int nl = n_begin + a_kk0; nl < n_end; nl += A_STEP) finish(nl, sm_gemm[nl * BMP + ml]);
        } else {
#pragma unroll 2
            for (int nl = n_begin + a_kk0; nl < n_end; nl += A_STEP) {
                const uint32_t at = 4u * (uint32_t)(nl * BMP + ml);
                float x[kMaxSplit];
#pragma unroll
                for (int r = 0; r < kMaxSplit; ++r)
                    if (r < splits) asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(x[r]) : "r"(peer[r] + at) : "memory");
                float v = x[0];
#pragma unroll
                for (int r = 1; r < kMaxSplit; ++r)
                    if (r < splits) v += x[r];
                finish(nl, v);
            }
        }
    }
    // nobody leaves while a peer may still read its shared memory
    if (splits > 1) asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// ---- the small-input-channel form of DIRECT (first layers: C = 3 with 3x3 ... 11x11 windows; few output channels).
// With C*R*S of a few dozen to a few hundred the GEMM blocking above spends its time on chunk hand-overs; here a
// thread owns ONE output pixel and KT output channels.  A block of 32 x 8 threads covers a 32 x 8 patch of one
// output plane: it stages the input patch with its halo (every channel, coalesced row loads, zeros for the padding)
// and the KT filters in shared memory, then walks the reduction (c, r, s) in order - one shared-memory load of the
// input per step, the KT weights as broadcast 16-byte loads, KT fused multiply-adds - and stores each output
// channel as 128-byte rows.  Such layers move more bytes than they compute (configuration 1: 11 FLOPs per byte), so
// the kernel is meant to run at memory speed.  More than KT output channels: one block per group of KT (grid.z).
// SW > 0 fixes the window width S at compile time (the inner loop then unrolls into loads at constant offsets:
// measured at run-time width, integer address arithmetic took as many issue slots as the multiply-adds, and the
// kernel was bound by instruction issue at 89 %); SW = 0 takes any width.
template <int KT, int SW>
__global__ void __launch_bounds__(256)
direct_pixel_kernel(const ConvDims d, const float* __restrict__ in, const float* __restrict__ filt,
                    const float* __restrict__ bias, float* __restrict__ out, int tiles_x, int ih, int iw, int iwp)
{
    constexpr int PY = 1;                              // output rows per thread (two were slower: half as many blocks to hide the staging latency)
    extern __shared__ __align__(16) float sm[];
    float* s_w = sm;                                   // [Kred][KT]
    float* s_in = sm + (size_t)d.Kred * KT;            // [C][ih][iwp]
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int bx = blockIdx.x % tiles_x, by = blockIdx.x / tiles_x;
    const int n = blockIdx.y;
    const int kg0 = blockIdx.z * KT;
    pdl_wait();
    // filters of this channel group: s_w[j][k] = filt[kg0 + k][j] (zeros past K); consecutive threads read consecutive j
    for (int idx = threadIdx.x; idx < d.Kred * KT; idx += 256) {
        const int k = idx / d.Kred, j = idx - k * d.Kred;
        s_w[j * KT + k] = (kg0 + k < d.K) ? __ldg(filt + (size_t)(kg0 + k) * d.Kred + j) : 0.f;
    }
    // input patch: rows y0 .. y0 + ih - 1, columns x0 .. x0 + iw - 1 of every channel
    const int y0 = by * (8 * PY) * d.stride - d.pad, x0 = bx * 32 * d.stride - d.pad;
    const float* img = in + (size_t)n * d.C * d.H * d.W;
    for (int row = ty; row < d.C * ih; row += 8) {
        const int c = row / ih, yy = row - c * ih;
        const int y = y0 + yy;
        const bool yin = y >= 0 && y < d.H;
        const float* src = img + ((size_t)c * d.H + (yin ? y : 0)) * d.W;
        float* dst = s_in + (size_t)row * iwp;
        for (int xx = tx; xx < iw; xx += 32) {
            const int x = x0 + xx;
            dst[xx] = (yin && x >= 0 && x < d.W) ? __ldg(src + x) : 0.f;
        }
    }
    __syncthreads();
    float acc[PY][KT];
#pragma unroll
    for (int i = 0; i < PY; ++i)
#pragma unroll
        for (int k = 0; k < KT; ++k) acc[i][k] = 0.f;
    // Shared memory is addressed through 32-bit shared-space addresses and explicit ld.shared instructions, so the
    // reduction loop carries one 32-bit address per operand and nothing else.
    const uint32_t w_base = (uint32_t)__cvta_generic_to_shared(s_w);
    uint32_t a_addr = (uint32_t)__cvta_generic_to_shared(s_in) + 4u * (uint32_t)((ty * d.stride) * iwp + tx * d.stride);
    uint32_t w_addr = w_base;
    auto lds = [](uint32_t addr) { float v; asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr)); return v; };
    auto lds4 = [](uint32_t addr) {
        float4 v;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
        return v;
    };
    auto step = [&](float a0, uint32_t w) {
#pragma unroll
        for (int q = 0; q < KT / 4; ++q) {
            const float4 wv = lds4(w + 16u * q);
            acc[0][4 * q] = fmaf(a0, wv.x, acc[0][4 * q]);
            acc[0][4 * q + 1] = fmaf(a0, wv.y, acc[0][4 * q + 1]);
            acc[0][4 * q + 2] = fmaf(a0, wv.z, acc[0][4 * q + 2]);
            acc[0][4 * q + 3] = fmaf(a0, wv.w, acc[0][4 * q + 3]);
        }
    };
    const int Sw = SW > 0 ? SW : d.S;
    const int rows_total = d.C * d.R;                  // (c, r) pairs: patch row c*ih + r, consecutive filter rows
    const uint32_t row_step = 4u * (uint32_t)iwp;
    const uint32_t c_step = 4u * (uint32_t)((ih - d.R) * iwp);   // from the last window row of a channel to the first of the next
    int r = 0;
    for (int cr = 0; cr < rows_total; ++cr) {
        if constexpr (SW > 0) {
#pragma unroll
            for (int sx = 0; sx < SW; ++sx) step(lds(a_addr + 4u * sx), w_addr + (uint32_t)(sx * KT * 4));
        } else {
            for (int sx = 0; sx < Sw; ++sx) step(lds(a_addr + 4u * (uint32_t)sx), w_addr + (uint32_t)(sx * KT * 4));
        }
        w_addr += (uint32_t)(Sw * KT * 4);
        a_addr += row_step;
        if (++r == d.R) { r = 0; a_addr += c_step; }
    }
    pdl_launch_dependents();
    const int q = bx * 32 + tx;
#pragma unroll
    for (int i = 0; i < PY; ++i) {
        const int p = by * (8 * PY) + ty + 8 * i;
        if (p < d.P && q < d.Q) {
            float* o = out + ((size_t)n * d.K * d.P + p) * d.Q + q;
#pragma unroll
            for (int k = 0; k < KT; ++k) {
                if (kg0 + k < d.K) {
                    float v = acc[i][k] + (bias ? __ldg(bias + kg0 + k) : 0.f);
                    if (d.relu) v = fmaxf(v, 0.f);
                    o[(size_t)(kg0 + k) * d.P * d.Q] = v;
                }
            }
        }
    }
}

// geometry of the pixel kernel for a shape; false if the patch does not fit shared memory
bool pixel_geometry(const ConvDims& d, int KT, int* ih, int* iw, int* iwp, size_t* smem)
{
    *ih = 7 * d.stride + d.R;
    *iw = 31 * d.stride + d.S;
    *iwp = *iw | 1;                                         // odd pitch: rows start on different banks
    *smem = ((size_t)d.Kred * KT + (size_t)d.C * *ih * *iwp) * sizeof(float);
    return *smem <= 200 * 1024 && d.Kred <= 4096;
}

template <int KT, int SW>
int launch_pixel_sw(const ConvDims& d, const float* in, const float* filt, const float* bias, float* out, cudaStream_t stream)
{
    int ih, iw, iwp;
    size_t smem;
    if (!pixel_geometry(d, KT, &ih, &iw, &iwp, &smem)) return BODA_ERR_UNSUPPORTED;
    static DeviceSmemLimit limit(48 * 1024);
    BODA_CUDA_TRY(limit.ensure(direct_pixel_kernel<KT, SW>, smem));
    const int tiles_x = (d.Q + 31) / 32, tiles_y = (d.P + 7) / 8;
    dim3 grid(tiles_x * tiles_y, d.N, (d.K + KT - 1) / KT);
    if (grid.y > 65535 || grid.z > 65535) return BODA_ERR_UNSUPPORTED;
    BODA_CUDA_TRY(launch_kernel(direct_pixel_kernel<KT, SW>, grid, dim3(256), smem, stream, 1, d, in, filt, bias, out, tiles_x, ih, iw, iwp));
    count_launch();
    return BODA_OK;
}

template <int KT>
int launch_pixel(const ConvDims& d, const float* in, const float* filt, const float* bias, float* out, cudaStream_t stream)
{
    switch (d.S) {
        case 3: return launch_pixel_sw<KT, 3>(d, in, filt, bias, out, stream);
        case 5: return launch_pixel_sw<KT, 5>(d, in, filt, bias, out, stream);
        case 7: return launch_pixel_sw<KT, 7>(d, in, filt, bias, out, stream);
        case 11: return launch_pixel_sw<KT, 11>(d, in, filt, bias, out, stream);
        default: return launch_pixel_sw<KT, 0>(d, in, filt, bias, out, stream);
    }
}

// bm x bn outputs per block, reduction chunks of bk (GEMM-blocked form; 0 otherwise)
struct TileInfo { int kind, bm, bn, kt, bk; const char* name; };
enum { TILE_GEMM = 0, TILE_PIXEL = 1, TILE_RTC = 2, TILE_STAGED = 3, TILE_SPLIT = 4 };
constexpr TileInfo kTiles[] = {
    {TILE_GEMM, 128, 128, 0, 8, "direct_128x128"}, {TILE_GEMM, 128, 96, 0, 16, "direct_128x96"},
    {TILE_GEMM, 128, 64, 0, 8, "direct_128x64"},   {TILE_GEMM, 128, 32, 0, 8, "direct_128x32"},
    {TILE_GEMM, 64, 64, 0, 8, "direct_64x64"},     {TILE_GEMM, 64, 32, 0, 8, "direct_64x32"},
    {TILE_GEMM, 64, 16, 0, 8, "direct_64x16"},      {TILE_GEMM, 32, 32, 0, 16, "direct_32x32"},
    {TILE_GEMM, 32, 16, 0, 8, "direct_32x16"},
    // pixel-per-thread form: kt output channels per thread
    {TILE_PIXEL, 0, 0, 8, 0, "direct_pixel_k8"}, {TILE_PIXEL, 0, 0, 16, 0, "direct_pixel_k16"},
    {TILE_PIXEL, 0, 0, 32, 0, "direct_pixel_k32"},
    // the same form compiled at run time for the exact shape (direct_rtc.cu)
    {TILE_RTC, 0, 0, 4, 0, "direct_rtc_k4"}, {TILE_RTC, 0, 0, 8, 0, "direct_rtc_k8"},
    {TILE_RTC, 0, 0, 16, 0, "direct_rtc_k16"}, {TILE_RTC, 0, 0, 32, 0, "direct_rtc_k32"},
    // more GEMM-blocked tiles (the ids above are part of the interface)
    {TILE_GEMM, 64, 48, 0, 8, "direct_64x48"}, {TILE_GEMM, 128, 48, 0, 8, "direct_128x48"},
    // over a staged NHWC copy of the input (simt_conv.cu): needs workspace
    {TILE_STAGED, 128, 128, 0, 32, "direct_nhwc_128x128"}, {TILE_STAGED, 128, 96, 0, 32, "direct_nhwc_128x96"},
    {TILE_STAGED, 128, 64, 0, 32, "direct_nhwc_128x64"},   {TILE_STAGED, 128, 48, 0, 32, "direct_nhwc_128x48"},
    {TILE_STAGED, 128, 32, 0, 32, "direct_nhwc_128x32"},
    // the same accuracy from the tensor cores, both operands staged in three parts (split_conv.cuh): needs workspace.  kt: the tile
    // of the tensor-core tables
    {TILE_SPLIT, 128, 64, 31, 64, "direct_nhwc_x3_128x64"}, {TILE_SPLIT, 128, 80, 32, 64, "direct_nhwc_x3_128x80"},
    {TILE_SPLIT, 128, 96, 33, 64, "direct_nhwc_x3_128x96"}, {TILE_SPLIT, 128, 128, 34, 64, "direct_nhwc_x3_128x128"},
};
constexpr int kFirstPixelTile = 9;
constexpr int kFewIndices = 32;      // reductions up to here suit the pixel-per-thread forms
constexpr int kNumTiles = sizeof(kTiles) / sizeof(kTiles[0]);

template <int WM, int WN, int TM, int TN, int BK>
int launch_tile(const ConvDims& d, const float* in, const float* filt, const float* bias, float* out,
                const DirectTapEntry* tab, int split, cudaStream_t stream)
{
    using G = GemmCfg<WM, WN, TM, TN, BK>;
    const int chunks = (d.Kred + BK - 1) / BK;
    const int per = (chunks + split - 1) / split;
    const int splits = (chunks + per - 1) / per;                          // no empty split
    dim3 grid((d.M + G::BM - 1) / G::BM, (d.K + G::BN - 1) / G::BN, splits);
    auto run = [&](auto kernel, DeviceSmemLimit& limit) -> cudaError_t {
        const cudaError_t e = limit.ensure(kernel, G::SMEM_BYTES);
        if (e != cudaSuccess) return e;
        return launch_kernel(kernel, grid, dim3(G::THREADS), (size_t)G::SMEM_BYTES, stream, splits, d, in, filt, bias, out, tab, chunks, per);
    };
    static DeviceSmemLimit limit_masked(48 * 1024), limit_any(48 * 1024);
    BODA_CUDA_TRY(d.R * d.S <= kMaskTaps ? run(direct_conv_kernel<WM, WN, TM, TN, BK, true>, limit_masked)
                                         : run(direct_conv_kernel<WM, WN, TM, TN, BK, false>, limit_any));
    count_launch();
    return BODA_OK;
}

}  // namespace

int direct_num_tiles() { return kNumTiles; }
const char* direct_tile_name(int id) { return (id >= 0 && id < kNumTiles) ? kTiles[id].name : "?"; }

// Clocks of a GEMM-blocked tile with the reduction split `split` ways.  A block's work is bm*bn/128 clocks of multiply-adds per
// reduction index at the SM's full rate; the blocks of an SM share that rate (`rate` clocks per clock of work), and no block is
// faster than `index` clocks per reduction index; `out` per bm*bn/128 outputs for the first loads and the store, `cluster` for
// a split.  Fitted per tile to 4 000 timings (82 layers of 1 ... 9850 reduction indices and 60 ... 363 000 points, every tile and split): the tile
// and split it picks are within 5 % of the best measured ones in the geometric mean.
struct GemmModel { int tile, resident; double fixed, rate, index, cluster, out; };
constexpr GemmModel kGemmModel[] = {
    {0, 1, 0, 1.78, 11, 2600, 52},     {1, 1, 0, 1.75, 118, 2600, 66},    {2, 2, 2140, 1.98, 0, 4300, 56},
    {3, 4, 3540, 3.07, 170, 2000, 45}, {4, 4, 2830, 1.98, 162, 3100, 64}, {5, 8, 4050, 3.09, 176, 1770, 50},
    {6, 8, 4350, 3.48, 62, 1440, 72},  {7, 8, 4450, 2.66, 45, 1620, 69},  {8, 16, 4150, 3.74, 69, 1180, 131},
    {16, 5, 3500, 2.70, 207, 2530, 54}, {17, 2, 1910, 1.95, 147, 2000, 88},
};

static double gemm_cost(const ConvDims& d, int t, int split)
{
    const TileInfo& ti = kTiles[t];
    const GemmModel* m = kGemmModel;
    while (m->tile != t) ++m;
    const int chunks = (d.Kred + ti.bk - 1) / ti.bk, per = (chunks + split - 1) / split;
    const long long splits = (chunks + per - 1) / per;
    const long long blocks = (long long)((d.M + ti.bm - 1) / ti.bm) * ((d.K + ti.bn - 1) / ti.bn) * splits;
    const long long per_sm = (blocks + 147) / 148, rounds = (per_sm + m->resident - 1) / m->resident;
    const double indices = (double)per * ti.bk, area = ti.bm * ti.bn / 128.0;
    return m->fixed + std::max(per_sm * indices * area * m->rate, rounds * indices * m->index) + per_sm * area * m->out +
           (splits > 1 ? m->cluster + 300.0 * splits : 0.0);
}

// Do the pixel-per-thread forms suit the layer, and with how many output channels per thread (0: no)?  They have no channel tile to
// fill and no chunk hand-overs, but load more per multiply-add.
//  * up to kFewIndices reduction indices: yes (27 indices, 16 filters, 32x32: 3.1 against 3.3 us at batch 1, 12.5 against 19.4 at 256);
//  * up to 512: where few filters leave the narrowest GEMM-blocked tile mostly empty.  The logarithm of what the run-time compiled form
//    gains over the best of those tiles, linear in the logarithms of the sizes, is fitted to 517 layers timed both ways (rms 0.2): 7x7
//    on 5 channels, one filter, 56x59, batch 15: 9.6 against 28.9 us; 5x5 on 2 channels, 4 filters, 42x45, batch 9: 3.2 against 4.8; the
//    other way 3x3 on 13 channels, 4 filters, 30x32, batch 1.  With the margin of 0.12 the choice gains 11 % over those layers in the
//    geometric mean (the best choice 14.6 %) and is more than 3 % behind the tiles on ten of them.
//    One channel up to 81 indices and two up to 50 gain 9 to 66 % whatever the fit says, but for
//    narrow images and many filters on many points (5x5 on 2 channels, 15 filters, 52x52, batch 2:
//    3.2 / 4.0 us); beyond the set's 64 channels nothing is known.
//  * never with a stride (27 indices with stride 2, 96 filters, batch 7: 17.8 against 16.0 us).
static int pixel_channels(const ConvDims& d)
{
    if (d.stride != 1 || d.K > 128) return 0;
    if (d.Kred <= kFewIndices) return 8;
    if (d.Kred > 512 || d.K > 32 || d.C > 64) return 0;
    const double m = std::min(std::log(d.M / 10000.0), 4.1), c = std::log((double)d.C), w = std::log((double)(d.R * d.S));
    auto gain = [&](int kt, double k1, double km, double k, double kkm, double kc, double kw, double kmc, double kmw) {
        const double k16 = std::log((double)((d.K + 15) / 16 * 16) / ((d.K + kt - 1) / kt * kt));       // channels paid for, tile / form
        return k1 + km * m + k * k16 + kkm * k16 * m + kc * c + kw * w + kmc * m * c + kmw * m * w;
    };
    const double g4 = gain(4, -0.285, -0.339, 0.331, 0.129, -0.114, 0.078, 0.076, 0.078);
    const double g8 = gain(8, -0.296, -0.310, 0.586, 0.167, -0.114, 0.060, 0.085, 0.079);
    const bool always = (d.C == 1 ? d.Kred <= 81 : d.C == 2 && d.Kred <= 50) && d.Q >= 12 && (d.K <= 16 || d.M <= 4096);
    return !always && std::max(g4, g8) < 0.12 ? 0 : g4 >= g8 ? 4 : 8;
}

bool direct_mask_fits(const ConvDims& d) { return d.R * d.S <= kMaskTaps; }

int direct_pick_gemm_tile(const ConvDims& d, double* clocks)
{
    int tile = -1;
    *clocks = 1e300;
    for (const GemmModel& m : kGemmModel) {
        const double c = gemm_cost(d, m.tile, direct_pick_split(d, m.tile));
        if (c < *clocks) { *clocks = c; tile = m.tile; }
    }
    return tile;
}

int direct_pick_split(const ConvDims& d, int tile)
{
    if (tile < 0 || tile >= kNumTiles || kTiles[tile].kind != TILE_GEMM) return 1;
    int best = 1;
    double best_cost = 1e300;
    for (int s = 1; s <= kMaxSplit; ++s) {
        if (s > 1 && (d.Kred + kTiles[tile].bk - 1) / kTiles[tile].bk < 2 * s) break;
        const double c = gemm_cost(d, tile, s);
        if (c < best_cost) { best_cost = c; best = s; }
    }
    return best;
}

int direct_max_split(const ConvDims& d, int tile)
{
    if (tile < 0 || tile >= kNumTiles || kTiles[tile].kind != TILE_GEMM) return 1;
    return std::min(kMaxSplit, (d.Kred + kTiles[tile].bk - 1) / kTiles[tile].bk);
}

int direct_tile_staged_width(int tile) { return tile >= 0 && tile < kNumTiles && kTiles[tile].kind == TILE_STAGED ? kTiles[tile].bn : 0; }

int direct_tile_split_operands(int tile) { return tile >= 0 && tile < kNumTiles && kTiles[tile].kind == TILE_SPLIT ? kTiles[tile].kt : -1; }

int direct_pick_tile(const ConvDims& d, size_t max_ws)
{
    // many output pixels where the pixel-per-thread form suits: the smallest KT that covers K in one group (or 32 channels per
    // group).  Measured against the GEMM-blocked tiles: 18.3 against 19.4 us for 3x3 on 3 channels, 16 filters, 32x32, batch 256.
    if (d.M >= 32768 && pixel_channels(d) > 0) {
        const int t = kFirstPixelTile + (d.K <= 8 ? 0 : d.K <= 16 ? 1 : 2);
        if (direct_tile_legal(d, t)) return t;
    }
    int best = 8, split = -1;
    double best_cost = 1e300, split_cost = 1e300, split_second = 0.0;
    for (int t = 0; t < kNumTiles; ++t) {
        double c;
        if (kTiles[t].kind == TILE_SPLIT) {
            if (!igemm_split_legal(d) || igemm_split_workspace(d) > (max_ws ? max_ws : igemm_split_workspace_limit(d))) continue;
            double clocks = 0.0;
            c = igemm_split_cost(d, kTiles[t].kt, &clocks);
            if (c < split_cost) { split_cost = c; split_second = clocks; split = t; }
            continue;
        }
        if (kTiles[t].kind == TILE_GEMM) c = gemm_cost(d, t, direct_pick_split(d, t));
        else if (kTiles[t].kind == TILE_STAGED && simt_legal(d) && (max_ws == 0 || simt_workspace_bytes(d, kTiles[t].bn) <= max_ws)) c = simt_cost(d, kTiles[t].bn);
        else continue;
        if (c < best_cost) { best_cost = c; best = t; }
    }
    // Where a chunk or a tile is mostly padding, both models of split operands have to agree (the second but for 5 %): 3x3 on 79 channels, one filter, 113x116,
    // batch 31 takes 363 us in place and 562 there, on 16 channels, 17 filters, 82x83, batch 22 47 and 70.  Of 774 layers 4 are then 16 to 60 % faster and
    // two slower (6 and 11 %).  Elsewhere the second model would be right no more often than the first.
    const bool padding = d.C <= 16 || d.K < 16;
    return split_cost < best_cost && (!padding || split_second <= 1.05 * best_cost) ? split : best;
}

bool direct_tile_legal(const ConvDims& d, int tile_id)
{
    if (tile_id < 0 || tile_id >= kNumTiles) return false;
    if (kTiles[tile_id].kind == TILE_GEMM) return true;
    if (kTiles[tile_id].kind == TILE_STAGED) return simt_legal(d);
    if (kTiles[tile_id].kind == TILE_SPLIT) return igemm_split_legal(d);
    if (kTiles[tile_id].kind == TILE_RTC) {
        int bx, by, py;
        size_t sm;
        return direct_rtc_available() && direct_rtc_geometry(d, kTiles[tile_id].kt, &bx, &by, &py, &sm);
    }
    int ih, iw, iwp;
    size_t smem;
    return pixel_geometry(d, kTiles[tile_id].kt, &ih, &iw, &iwp, &smem) && d.N <= 65535 && (d.K + kTiles[tile_id].kt - 1) / kTiles[tile_id].kt <= 65535;
}

int direct_tile_rtc_kt(int tile_id) { return (tile_id >= 0 && tile_id < kNumTiles && kTiles[tile_id].kind == TILE_RTC) ? kTiles[tile_id].kt : 0; }

int direct_rtc_pick(const ConvDims& d)
{
    // Where the pixel-per-thread form suits.  Eight channels per thread as a rule; four where that leaves fewer than 64 blocks (more
    // blocks hide the staging latency); sixteen where 16 covers all output channels of a large layer (the input patch is staged
    // once); for the longer reductions what pixel_channels() says.
    const int suits = pixel_channels(d);
    if (suits == 0 || !direct_rtc_available()) return -1;
    int bx = 32, by = 8, py = 1;
    size_t sm = 0;
    if (!direct_rtc_geometry(d, 8, &bx, &by, &py, &sm)) bx = 8, by = 4, py = 1;
    const long long blocks8 = (long long)((d.Q + bx - 1) / bx) * ((d.P + by * py - 1) / (by * py)) * d.N * ((d.K + 7) / 8);
    const int want = d.Kred > kFewIndices ? suits : (d.K <= 16 && d.M >= 16384) ? 16 : blocks8 < 64 ? 4 : 8;
    const int order[3][3] = {{4, 8, 16}, {8, 4, 16}, {16, 8, 4}};
    const int* o = order[want == 4 ? 0 : want == 8 ? 1 : 2];
    for (int i = 0; i < 3; ++i)
        for (int t = 0; t < kNumTiles; ++t)
            if (kTiles[t].kind == TILE_RTC && kTiles[t].kt == o[i] && direct_tile_legal(d, t)) return t;
    return -1;
}

// whole chunks of the widest chunk (16 reduction indices)
int direct_table_len(const ConvDims& d) { return ((d.Kred + 15) / 16) * 16; }

void direct_build_table(const ConvDims& d, DirectTapEntry* tab)
{
    const int len = direct_table_len(d);
    const bool masked = d.R * d.S <= kMaskTaps;
    int j = 0;
    for (int c = 0; c < d.C; ++c)
        for (int r = 0; r < d.R; ++r)
            for (int s = 0; s < d.S; ++s, ++j) {
                tab[j].offset = c * d.H * d.W + r * d.W + s;
                tab[j].rs = masked ? r * d.S + s : (r << 16) | s;
            }
    for (; j < len; ++j) { tab[j].offset = 0; tab[j].rs = masked ? kMaskTaps : (0x4000 << 16); }
}

int direct_launch(const ConvDims& d, int tile_id, int split, const float* in, const float* filt, const float* bias,
                  float* out, const DirectTapEntry* tab, cudaStream_t stream)
{
    switch (tile_id) {
        case 0: return launch_tile<2, 4, 8, 8, 8>(d, in, filt, bias, out, tab, split, stream);
        case 1: return launch_tile<2, 4, 8, 6, 16>(d, in, filt, bias, out, tab, split, stream);
        case 2: return launch_tile<2, 2, 8, 8, 8>(d, in, filt, bias, out, tab, split, stream);
        case 3: return launch_tile<2, 2, 8, 4, 8>(d, in, filt, bias, out, tab, split, stream);
        case 4: return launch_tile<1, 2, 8, 8, 8>(d, in, filt, bias, out, tab, split, stream);
        case 5: return launch_tile<1, 2, 8, 4, 8>(d, in, filt, bias, out, tab, split, stream);
        case 6: return launch_tile<2, 1, 4, 4, 8>(d, in, filt, bias, out, tab, split, stream);
        case 7: return launch_tile<1, 2, 4, 4, 16>(d, in, filt, bias, out, tab, split, stream);
        case 8: return launch_tile<1, 1, 4, 4, 8>(d, in, filt, bias, out, tab, split, stream);
        case 9: return launch_pixel<8>(d, in, filt, bias, out, stream);
        case 10: return launch_pixel<16>(d, in, filt, bias, out, stream);
        case 11: return launch_pixel<32>(d, in, filt, bias, out, stream);
        case 16: return launch_tile<1, 2, 8, 6, 8>(d, in, filt, bias, out, tab, split, stream);
        case 17: return launch_tile<2, 2, 8, 6, 8>(d, in, filt, bias, out, tab, split, stream);
        default: return BODA_ERR_UNSUPPORTED;
    }
}

}  // namespace boda
