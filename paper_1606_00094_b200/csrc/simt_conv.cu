// DIRECT over a staged input: FP32 implicit-GEMM convolution on the CUDA cores, fed by TMA.
//
// Bound: the FP32 pipe (128 multiply-adds per clock and SM).  The gather of the GEMM-blocked kernel in direct_conv.cu spends
// more issue slots on addresses, bounds and copies than on multiply-adds; here a staging kernel writes the input once as NHWC
// rows (fp32 as it is) and the copy engine does all of the gather: TMA im2col loads bring 128 output points x 32 channels per
// step, tiled loads the matching filter rows, both as 128-byte rows with the 128-byte swizzle.  Eight warps do nothing but
// shared-memory loads and packed multiply-adds (__ffma2_rn, each half rounds like fmaf): an accumulator's two halves sum the
// even and the odd channels, so the four channels of a 16-byte load are two ready operands and nothing moves between registers.
//
// Persistent, with an even split of the work: tiles that fill whole rounds of the SMs are computed whole; the rest is one run of
// reduction steps cut into as many equal pieces as there are CTAs, whatever the tile boundaries.  A piece that covers a tile only
// in part writes its sums to the workspace, and a second kernel adds the pieces of such tiles in order (every run gives the
// same bits), adds the bias, applies ReLU and stores.
//
// Measured, 3x3 on 256 channels, 384 filters, 13x13, batch 20 (6.0 GFLOP, 80 us at the pipe's 74 TFLOP/s): 499 us on the
// GEMM-blocked kernel as it was (4-byte gather, 32x32 tiles), 171 us on its packed and split successor, 136 us here (staging
// of both operands, the main kernel's 126, sums 5): the main kernel runs at 64 % of the pipe's peak rate.  16 warps of 8 x 4 pairs instead of 8 of 8 x 8
// took 159 us (more operand loads per multiply-add), two CTAs per SM with plain fmaf 174 us (register-bank conflicts).
#include <cuda.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <new>

#define BODA_WAIT_KERNEL_ID KERNEL_ID_SIMT
#include "simt_conv.h"
#include "stage.h"
#include "tc_ptx.cuh"

namespace boda {
namespace {

using namespace tc;

constexpr int BM = 128, BKC = 32;
constexpr int A_STAGE_BYTES = BM * 128;
constexpr int kWarps = 8;                                // two a scheduler: 255 registers a thread hold 8 x 8 accumulator pairs
constexpr int kThreads = 32 * kWarps;
constexpr int kMinSteps = 4;                             // reduction steps a CTA is worth starting for

struct SimtParams {
    int M, K, Q, PQ, stride, pad, S;
    int cchunks, last_groups;                            // 32-channel chunks; 4-channel groups of the last one that hold data
    int steps;                                           // reduction steps per tile: taps * cchunks
    int tiles_n, whole_tiles, cut_tiles;                 // tiles computed whole, then tiles cut into equal pieces
    const float* bias;
    float* out;
    float* partial;                                      // two slots of [BN][128] per CTA
    int relu;
    int* status;
    int tx_extra;                                        // test hook: bytes the first stage of CTA 0 expects and never gets
};

template <int WM, int WN, int TM, int TN>
struct Cfg {
    static_assert(WM * WN == kWarps && 8 * WM * TM == BM, "the warps cover the 128 points");
    static constexpr int BN = 4 * WN * TN;
    static constexpr int B_STAGE_BYTES = BN * 128;
    static constexpr int STAGE_BYTES = A_STAGE_BYTES + B_STAGE_BYTES;
    static constexpr int STAGES = (200 * 1024) / STAGE_BYTES > 8 ? 8 : (200 * 1024) / STAGE_BYTES;
    static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 256;
};

// first step of CTA b's share of `total` steps
__device__ __forceinline__ long long share_begin(long long total, int b, int ctas) { return total * b / ctas; }

// A CTA's work, piece by piece: steps [i0, i1) of a tile; slot < 0 for a tile computed whole.
struct Walk {
    int whole_next;
    long long cur, s0, s1;
    int tile, i0, i1, slot;
    __device__ __forceinline__ void start(const SimtParams& p)
    {
        const long long total = (long long)p.cut_tiles * p.steps;
        whole_next = (int)blockIdx.x;
        s0 = cur = share_begin(total, (int)blockIdx.x, (int)gridDim.x);
        s1 = share_begin(total, (int)blockIdx.x + 1, (int)gridDim.x);
    }
    __device__ __forceinline__ bool next(const SimtParams& p)
    {
        if (whole_next < p.whole_tiles) {
            tile = whole_next; i0 = 0; i1 = p.steps; slot = -1;
            whole_next += (int)gridDim.x;
            return true;
        }
        if (cur >= s1) return false;
        const int t = (int)(cur / p.steps);
        i0 = (int)(cur - (long long)t * p.steps);
        i1 = (int)min((long long)p.steps, i0 + (s1 - cur));
        slot = (i0 == 0 && i1 == p.steps) ? -1 : 2 * (int)blockIdx.x + (cur != s0 ? 1 : 0);
        tile = p.whole_tiles + t;
        cur += i1 - i0;
        return true;
    }
};

template <int WM, int WN, int TM, int TN>
__global__ void __launch_bounds__(kThreads, 1)
simt_conv_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, const SimtParams p)
{
    using G = Cfg<WM, WN, TM, TN>;
    constexpr int BN = G::BN, STAGES = G::STAGES;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* const smem = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t full_bar = smem_base + STAGES * G::STAGE_BYTES, empty_bar = full_bar + 8 * STAGES;
    __shared__ volatile int s_abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    pdl_launch_dependents();
    if (threadIdx.x == 0) {
        s_abort = 0;
        for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar + 8 * s, 1); mbar_init(empty_bar + 8 * s, kWarps); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        prefetch_tensormap(&map_a);
        prefetch_tensormap(&map_b);
    }
    __syncthreads();
    pdl_wait();

    // ---------------- loads: one lane of warp 0 keeps STAGES - 2 steps in flight ahead of its own warp's arithmetic, so that the
    // stage it refills was left two steps ago and the other warps have had a whole step to leave it too
    constexpr int AHEAD = STAGES - 2;
    static_assert(AHEAD >= 1, "the ring holds a step ahead");
    const bool loader = threadIdx.x == 0;
    Walk lw;
    uint32_t l_stage = 0, l_par = 1;
    int l_i = 0, l_cx = 0, l_tap = 0, l_r = 0, l_s = 0, l_w0 = 0, l_h0 = 0, l_n0 = 0, l_k0 = 0;
    bool l_more = false;
    auto load_piece = [&]() {
        l_more = lw.next(p);
        if (!l_more) return;
        const int tm = lw.tile / p.tiles_n, m0 = tm * BM;
        l_k0 = (lw.tile - tm * p.tiles_n) * BN;
        l_n0 = m0 / p.PQ;
        const int rem = m0 - l_n0 * p.PQ, p0 = rem / p.Q, q0 = rem - p0 * p.Q;
        l_w0 = q0 * p.stride - p.pad; l_h0 = p0 * p.stride - p.pad;
        l_i = lw.i0;
        l_tap = l_i / p.cchunks; l_cx = (l_i - l_tap * p.cchunks) * BKC;
        l_r = l_tap / p.S; l_s = l_tap - l_r * p.S;
    };
    auto load_step = [&]() {          // false: a wait ran out
        if (!l_more) return true;
        if (!mbar_wait(empty_bar + 8 * l_stage, l_par, &s_abort, p.status, 51)) return false;
        const uint32_t dst = smem_base + l_stage * G::STAGE_BYTES, fb = full_bar + 8 * l_stage;
        mbar_expect_tx(fb, G::STAGE_BYTES);
        tma_load_im2col_4d(dst, &map_a, fb, l_cx, l_w0, l_h0, l_n0, (uint16_t)l_s, (uint16_t)l_r);
        tma_load_3d(dst + A_STAGE_BYTES, &map_b, fb, l_cx, l_k0, l_tap);
        if (++l_stage == (uint32_t)STAGES) { l_stage = 0; l_par ^= 1u; }
        l_cx += BKC;
        if (l_cx == p.cchunks * BKC) { l_cx = 0; ++l_tap; if (++l_s == p.S) { l_s = 0; ++l_r; } }
        if (++l_i == lw.i1) load_piece();
        return true;
    };
    if (loader) {
        if (p.tx_extra && blockIdx.x == 0)
            asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" :: "r"(full_bar), "r"(p.tx_extra) : "memory");
        lw.start(p);
        load_piece();
        for (int i = 0; i < AHEAD; ++i) (void)load_step();
    }

    // ---------------- arithmetic.  Lane bits 1, 3, 4 pick the point, bits 0, 2 the channel: lanes i and i^1 read
    // the same input row and lanes i and i^2 the same filter row, so that a 16-byte shared-memory load serves two quarter
    // warps at once (measured on the GEMM-blocked kernel: half the wavefronts).
    const int lane_m = ((lane >> 1) & 1) | ((lane >> 2) & 6), lane_n = (lane & 1) | ((lane >> 1) & 2);
    const int wm = warp % WM, wn = warp / WM;
    const int m_local = wm * 8 * TM + lane_m, n_local = wn * 4 * TN + lane_n;     // + 8*i, + 4*j
    uint32_t stage = 0, par = 0;
    Walk walk;
    walk.start(p);
    while (walk.next(p)) {
        const int tile = walk.tile, i0 = walk.i0, i1 = walk.i1, slot = walk.slot;
        float2 acc[TM][TN];
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) acc[i][j] = make_float2(0.f, 0.f);
        int chunk = i0 % p.cchunks;
        for (int it = i0; it < i1; ++it) {
            if (loader) (void)load_step();
            if (!mbar_wait(full_bar + 8 * stage, par, &s_abort, p.status, 52)) return;
            __syncwarp();                // the loading lane rejoins its warp
            const uint8_t* a_row = smem + stage * G::STAGE_BYTES + m_local * 128;
            const uint8_t* b_row = smem + stage * G::STAGE_BYTES + A_STAGE_BYTES + n_local * 128;
            const int groups = chunk + 1 == p.cchunks ? p.last_groups : 8;
#pragma unroll 1
            for (int g = 0; g < groups; ++g) {
                // 16-byte piece g of a row sits at piece g ^ (row & 7)
                const uint8_t* as = a_row + ((g ^ lane_m) << 4);
                const uint8_t* bs = b_row + ((g ^ lane_n) << 4);
                const uint8_t* bs4 = b_row + ((g ^ (lane_n + 4)) << 4);
                float4 a[TM];
#pragma unroll
                for (int i = 0; i < TM; ++i) a[i] = *reinterpret_cast<const float4*>(as + 1024 * i);
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    const float4 b = *reinterpret_cast<const float4*>(((j & 1) ? bs4 : bs) + 512 * j);
                    const float2 b01 = make_float2(b.x, b.y), b23 = make_float2(b.z, b.w);
#pragma unroll
                    for (int i = 0; i < TM; ++i) acc[i][j] = __ffma2_rn(make_float2(a[i].x, a[i].y), b01, acc[i][j]);
#pragma unroll
                    for (int i = 0; i < TM; ++i) acc[i][j] = __ffma2_rn(make_float2(a[i].z, a[i].w), b23, acc[i][j]);
                }
            }
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(empty_bar + 8 * stage) : "memory");
            if (++stage == (uint32_t)STAGES) { stage = 0; par ^= 1u; }
            if (++chunk == p.cchunks) chunk = 0;
        }
        if (slot >= 0) {
            float* dst = p.partial + (size_t)slot * (BM * BN) + m_local;
#pragma unroll
            for (int j = 0; j < TN; ++j)
#pragma unroll
                for (int i = 0; i < TM; ++i) dst[(n_local + 4 * j) * BM + 8 * i] = acc[i][j].x + acc[i][j].y;
            continue;
        }
        const int tm = tile / p.tiles_n, k0 = (tile - tm * p.tiles_n) * BN + n_local;
        float bias[TN];
#pragma unroll
        for (int j = 0; j < TN; ++j) bias[j] = (p.bias && k0 + 4 * j < p.K) ? __ldg(p.bias + k0 + 4 * j) : 0.f;
#pragma unroll
        for (int i = 0; i < TM; ++i) {
            const int m = tm * BM + m_local + 8 * i;
            if (m >= p.M) continue;
            const int n = m / p.PQ;
            float* o = p.out + ((size_t)n * p.K + k0) * p.PQ + (m - n * p.PQ);
#pragma unroll
            for (int j = 0; j < TN; ++j) {
                float v = acc[i][j].x + acc[i][j].y + bias[j];
                if (p.relu) v = fmaxf(v, 0.f);
                if (k0 + 4 * j < p.K) o[(size_t)(4 * j) * p.PQ] = v;
            }
        }
    }
}

// Sums the pieces of the cut tiles: block (tile, group of channels), a thread owns one point and has its channels' loads in
// flight together (bound: latency; a few pieces of 64 KB a tile, still in L2).
constexpr int kSumChannels = 8;
template <int BN>
__global__ void __launch_bounds__(BM)
simt_sum_kernel(const SimtParams p, int ctas)
{
    pdl_launch_dependents();
    pdl_wait();                  // in every block: a grid that ends without waiting would let the next one overtake the main kernel
    const int t = (int)blockIdx.x;
    const long long total = (long long)p.cut_tiles * p.steps, a = (long long)t * p.steps, e = a + p.steps;
    int b0 = (int)(a * ctas / total);
    while (share_begin(total, b0 + 1, ctas) <= a) ++b0;
    while (share_begin(total, b0, ctas) > a) --b0;
    if (share_begin(total, b0 + 1, ctas) >= e) return;                     // one CTA had all of it and has stored it
    int b1 = b0 + 1;                                                       // pieces: CTAs b0 .. b1 - 1
    while (b1 < ctas && share_begin(total, b1, ctas) < e) ++b1;
    const int tile = p.whole_tiles + t;
    const int tm = tile / p.tiles_n, k0 = (tile - tm * p.tiles_n) * BN;
    const int m = tm * BM + (int)threadIdx.x;
    const int n = m / p.PQ;
    // the first piece is its CTA's last one if the CTA began in an earlier tile; the others are their CTAs' first ones
    const int first_slot = 2 * b0 + (share_begin(total, b0, ctas) < a ? 1 : 0);
    if (m >= p.M) return;
    const int c0 = (int)blockIdx.y * kSumChannels;
    const float* src = p.partial + (size_t)c0 * BM + threadIdx.x;
    float v[kSumChannels];
#pragma unroll
    for (int c = 0; c < kSumChannels; ++c) v[c] = __ldg(src + (size_t)first_slot * (BM * BN) + c * BM);
#pragma unroll 2
    for (int b = b0 + 1; b < b1; ++b)
#pragma unroll
        for (int c = 0; c < kSumChannels; ++c) v[c] += __ldg(src + (size_t)(2 * b) * (BM * BN) + c * BM);
    float* o = p.out + ((size_t)n * p.K + k0 + c0) * p.PQ + (m - n * p.PQ);
#pragma unroll
    for (int c = 0; c < kSumChannels; ++c) {
        if (k0 + c0 + c >= p.K) break;
        float y = v[c] + (p.bias ? __ldg(p.bias + k0 + c0 + c) : 0.f);
        if (p.relu) y = fmaxf(y, 0.f);
        o[(size_t)c * p.PQ] = y;
    }
}

constexpr int kSms = 148;

struct Schedule { int tiles_m, tiles_n, steps, ctas, whole, cut; };

Schedule schedule(const ConvDims& d, int bn, int sms)
{
    Schedule s;
    s.tiles_m = (d.M + BM - 1) / BM;
    s.tiles_n = (d.K + bn - 1) / bn;
    s.steps = d.R * d.S * ((d.C + BKC - 1) / BKC);
    const long long tiles = (long long)s.tiles_m * s.tiles_n;
    // whole rounds stay uncut except the last full one, which is cut together with the remainder: a CTA then has between one
    // and two tiles' worth of cut work.  (With fewer CTAs than SMs, where a tile has less than kMinSteps steps, it has more.)  At
    // most two of its pieces are partial, its first and its last; what lies between is whole tiles.
    const long long rounds = tiles / sms;
    s.whole = tiles % sms == 0 ? (int)tiles : (int)(rounds > 1 ? (rounds - 1) * sms : 0);
    s.cut = (int)(tiles - s.whole);
    s.ctas = (int)std::min<long long>(sms, std::max<long long>(1, s.whole > 0 ? sms : tiles * s.steps / kMinSteps));
    return s;
}

}  // namespace

struct SimtPlan {
    ConvDims d;
    int bn = 128, Cp = 32;
    Schedule s;
    float* d_wp = nullptr;
    size_t xp_bytes = 0;
    CUtensorMap map_a, map_b;
    const void* map_a_base = nullptr;
    int* d_status = nullptr;
    int tx_extra = 0;
};

bool simt_legal(const ConvDims& d)
{
    // limits of the im2col loads (window offsets and pads are small signed numbers)
    return d.R <= 11 && d.S <= 11 && d.stride <= 8 && d.pad <= 100 && d.P > 0 && d.Q > 0 && (long long)d.M * ((d.K + 31) / 32) <= 0x7fffffffLL;
}

static size_t staged_bytes(const ConvDims& d)
{
    const size_t Cp = (size_t)((d.C + BKC - 1) / BKC) * BKC;
    return ((size_t)d.N * d.H * d.W * Cp * 4 + 1023) & ~(size_t)1023;
}

size_t simt_workspace_bytes(const ConvDims& d, int bn)
{
    const Schedule s = schedule(d, bn, kSms);
    return staged_bytes(d) + (s.cut > 0 ? (size_t)2 * s.ctas * BM * bn * 4 : 0);
}

double simt_cost(const ConvDims& d, int bn)
{
    const Schedule s = schedule(d, bn, kSms);
    // fitted to the same timings as the GEMM-blocked tiles' model (rms 11 %)
    const int chunks = (d.C + BKC - 1) / BKC;
    const double steps = (double)s.whole / kSms * s.steps + (double)s.cut * s.steps / s.ctas;
    const double live = (double)((d.C + 3) / 4 * 4) / (chunks * BKC);        // part of the chunks that holds data
    const double filters = (double)d.K * d.R * d.S * (d.C + chunks * BKC) * 4;
    const double staging = ((double)d.N * d.C * d.H * d.W * 4 + (double)staged_bytes(d) + filters) / 1734.0;
    const double sums = s.cut == 0 ? 0.0 : 11400.0 + 518.0 * std::max(0.0, (double)s.ctas / s.cut - 1.0) + 2.0 * s.ctas * BM * bn * 4 / 3427.0;
    return staging + 9970.0 + steps * (32.0 * bn * live * 1.36 + 678.0) + sums;
}

int simt_plan_create(const ConvDims& d, int bn, int* d_status, SimtPlan** out)
{
    if (!simt_legal(d)) return BODA_ERR_UNSUPPORTED;
    int rc = load_driver_entry_points();
    if (rc != BODA_OK) return rc;
    SimtPlan* p = new (std::nothrow) SimtPlan();
    if (!p) return BODA_ERR_NOMEM;
    p->d = d;
    p->bn = bn;
    p->Cp = ((d.C + BKC - 1) / BKC) * BKC;
    p->d_status = d_status;
    p->tx_extra = test_tx_extra();
    if ((rc = upload_wait_limit()) != BODA_OK) { delete p; return rc; }
    p->s = schedule(d, bn, kSms);
    p->xp_bytes = staged_bytes(d);
    cudaError_t e = cudaMalloc(&p->d_wp, (size_t)d.R * d.S * d.K * p->Cp * 4);
    if (e != cudaSuccess) { simt_plan_destroy(p); return record_cuda_error(e, "FP32 plan allocation"); }
    const cuuint64_t dims[3] = {(cuuint64_t)p->Cp, (cuuint64_t)d.K, (cuuint64_t)(d.R * d.S)};
    const cuuint64_t strides[2] = {(cuuint64_t)p->Cp * 4, (cuuint64_t)d.K * p->Cp * 4};
    const cuuint32_t box[3] = {BKC, (cuuint32_t)bn, 1}, estr[3] = {1, 1, 1};
    const CUresult r = g_encode_tiled(&p->map_b, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, p->d_wp, dims, strides, box, estr,
                                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) { simt_plan_destroy(p); return record_cuda_error(cudaErrorInvalidValue, "cuTensorMapEncodeTiled (FP32 filters)"); }
    *out = p;
    return BODA_OK;
}

void simt_plan_destroy(SimtPlan* p)
{
    if (!p) return;
    if (p->d_wp) cudaFree(p->d_wp);
    delete p;
}

int simt_plan_kernels(const SimtPlan* p) { return p->s.cut > 0 ? 3 : 2; }

void simt_plan_describe(const SimtPlan* p, char* buf, size_t n)
{
    std::snprintf(buf, n, "grid=%d tiles=%dx%d cut=%d steps=%d", p->s.ctas, p->s.tiles_m, p->s.tiles_n, p->s.cut, p->s.steps);
}

namespace {

template <int WM, int WN, int TM, int TN>
int launch_width(SimtPlan* p, const SimtParams& prm, cudaStream_t stream)
{
    using G = Cfg<WM, WN, TM, TN>;
    static DeviceSmemLimit limit;
    BODA_CUDA_TRY(limit.ensure(simt_conv_kernel<WM, WN, TM, TN>, G::SMEM_BYTES));
    BODA_CUDA_TRY(launch_kernel(simt_conv_kernel<WM, WN, TM, TN>, dim3(p->s.ctas), dim3(kThreads), (size_t)G::SMEM_BYTES, stream, 1, p->map_a,
                                p->map_b, prm));
    count_launch();
    if (p->s.cut == 0) return BODA_OK;
    BODA_CUDA_TRY(launch_kernel(simt_sum_kernel<G::BN>, dim3(p->s.cut, G::BN / kSumChannels), dim3(BM), 0, stream, 1, prm, p->s.ctas));
    count_launch();
    return BODA_OK;
}

}  // namespace

int simt_launch(SimtPlan* p, const float* in, const float* filt, const float* bias, float* out, void* workspace, cudaStream_t stream,
                cudaEvent_t after_staging)
{
    const ConvDims& d = p->d;
    if (!workspace) return BODA_ERR_NOMEM;
    if (((uintptr_t)workspace & 255) != 0) return BODA_ERR_INVALID_ARG;
    if (!filt) return BODA_ERR_INVALID_ARG;
    // Both operands on every call: FP32 plans read the caller's filters anew each time, as the kernels that use them in place do.
    const StageInput x = {in, workspace, d.N, d.C, p->Cp, d.H * d.W};
    const StageFilters w = {filt, p->d_wp, d.K, d.C, p->Cp, d.R * d.S};
    int rc = stage_operands(STAGE_FP32, &x, &w, stream);
    if (rc != BODA_OK) return rc;
    if (p->map_a_base != workspace) {
        const cuuint64_t Cp = (cuuint64_t)p->Cp;
        const cuuint64_t dims[4] = {Cp, (cuuint64_t)d.W, (cuuint64_t)d.H, (cuuint64_t)d.N};
        const cuuint64_t strides[3] = {Cp * 4, (cuuint64_t)d.W * Cp * 4, (cuuint64_t)d.H * d.W * Cp * 4};
        const int lower[2] = {-d.pad, -d.pad}, upper[2] = {d.pad - (d.S - 1), d.pad - (d.R - 1)};
        const cuuint32_t estr[4] = {1, (cuuint32_t)d.stride, (cuuint32_t)d.stride, 1};
        const CUresult r = g_encode_im2col(&p->map_a, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, workspace, dims, strides, lower, upper, BKC, BM, estr,
                                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return record_cuda_error(cudaErrorInvalidValue, "cuTensorMapEncodeIm2col (FP32 input)");
        p->map_a_base = workspace;
    }
    if (after_staging) BODA_CUDA_TRY(cudaEventRecord(after_staging, stream));
    SimtParams prm;
    prm.M = d.M; prm.K = d.K; prm.Q = d.Q; prm.PQ = d.P * d.Q;
    prm.stride = d.stride; prm.pad = d.pad; prm.S = d.S;
    prm.cchunks = p->Cp / BKC;
    prm.last_groups = (d.C - BKC * (prm.cchunks - 1) + 3) / 4;
    prm.steps = p->s.steps;
    prm.tiles_n = p->s.tiles_n; prm.whole_tiles = p->s.whole; prm.cut_tiles = p->s.cut;
    prm.bias = bias; prm.out = out; prm.relu = d.relu; prm.status = p->d_status; prm.tx_extra = p->tx_extra;
    prm.partial = reinterpret_cast<float*>(static_cast<char*>(workspace) + p->xp_bytes);
    switch (p->bn) {
        case 128: return launch_width<2, 4, 8, 8>(p, prm, stream);
        case 96: return launch_width<2, 4, 8, 6>(p, prm, stream);
        case 64: return launch_width<2, 4, 8, 4>(p, prm, stream);
        case 48: return launch_width<4, 2, 4, 6>(p, prm, stream);
        case 32: return launch_width<4, 2, 4, 4>(p, prm, stream);
        default: return BODA_ERR_UNSUPPORTED;
    }
}

}  // namespace boda
