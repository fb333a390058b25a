// K1CONV and TCONV on pairs of SMs: the im2col kernel's operands (igemm_tf32.cu) with tcgen05.mma.cta_group::2, persistent.
//
// Two CTAs of a cluster share one output tile of 256 points x BN channels: each stages its own 128 points and HALF of the tile's
// filter rows, and one thread of the first CTA issues MMAs that read both CTAs' shared memory and write 128 rows into each
// CTA's tensor memory.  A CTA therefore fetches 128 + BN/2 rows per reduction step instead of 128 + BN for the same MMA time.
// The fetch is what bounds the one-CTA kernel below BN = 192: with every SM busy a step of 128 channels takes it 297 clocks for 256 of MMAs (L2 gives it 16.3 KB a
// clock in all, fitted; the pairs 13.7), a pair 265.
// The pairs are persistent (at most one CTA per SM walks the tiles) with two accumulators in tensor memory: a tile's epilogue
// and the pipeline's fill run under the next tile's main loop.
// Measured, one-CTA kernel / pairs of the same width: 5x5 on 96 channels, 256 filters, 27x27, fp16, batch 128 (115 GFLOP) 130 / 105 us (BN = 256), 153 / 123
// (128); 3x3 on 256 channels, 384 filters, 13x13, batch 128 73.3 / 63.1 (128), 70.9 / 65.6 (192).
// One round of few tiles stays with the one-CTA kernel (3x3, 13x13, batch 20: 16.8 / 17.6 us, BN = 96).
//
// Roles per CTA (416 threads): warp 0 = input tiles, warp 11 = filter tiles, warp 12 (first CTA) = byte counts of both CTAs, warp
// 1 = MMA issue (first CTA) and the tensor-memory allocation, warps 2..5 and 7..10 = epilogue.  Loads signal the first CTA's full
// barriers; tcgen05.commit releases a stage in both CTAs.  All loads are plain (no multicast).  Waits are bounded as elsewhere.
#pragma once

#include "tc_ptx.cuh"

namespace boda {
namespace pair {

using namespace tc;

constexpr int kThreads = 416;
constexpr int A_CHUNK_BYTES = 128 * 128;
constexpr int BOX_BYTES = 32 * 128;          // 32 rows x 32 channels: what an epilogue warp hands to the tensor store

struct PairParams {
    int M, stride, pad, S;
    int cchunks;                 // reduction chunks per tap (128 bytes of channels each)
    int last_ksteps;             // 32-byte MMA steps of a tap's last chunk that hold channels (1..4): the rest are padding and skipped
    int iters;                   // taps * cchunks
    int accs;                    // accumulators that a tile's stages take turns with (at most Cfg::ACCS, and the stages of a tile)
    int tiles_n, tiles_total;    // tiles are numbered point tile * tiles_n + channel tile
    const float* bias;
    OutSpec o;
    int* status;
    int tx_extra;                // test hook: bytes added to the expected size of the first stage of the first pair
    int b_early;                 // bound filters: their loads need not wait for the preceding kernel
    int out_tma;                 // staged output without padding rows or columns: boxes leave through the output tensor map
};

template <int BN> struct Cfg {
    static constexpr int B_ROWS = BN / 2;
    static constexpr int B_CHUNK_BYTES = B_ROWS * 128;
    // Reduction chunks per stage: a stage costs the issuing warp a wait, a vote and a commit besides its MMAs, so the narrower tiles put two
    // chunks in one.
    static constexpr int CPS = BN >= 256 ? 1 : 2;
    static constexpr int STAGE_BYTES = CPS * (A_CHUNK_BYTES + B_CHUNK_BYTES);
    static constexpr int STORE_BYTES = 8 * BOX_BYTES;
    static constexpr int STAGES = BN >= 256 ? 5 : (192 * 1024) / STAGE_BYTES;
    // Accumulators that a tile may have, taking the stages in turn; two tiles' worth fill tensor memory.  The tensor core truncates
    // an accumulator at every MMA, so the error of a sum grows with the MMAs that one accumulator takes: measured 1.6e-8 of the
    // result per MMA (1563 of them 2.5e-5).  Reading more than one back costs a short reduction up to 10 % (its epilogue does not
    // hide under the next tile), and a changing accumulator address the issue loop 1 to 2 %, so only the longer reductions have
    // them (PairParams::accs), in a form of the kernel of their own (MULTI).
    static constexpr int ACCS = BN <= 64 ? 4 : BN <= 128 ? 2 : 1;
    static_assert(2 * ACCS * BN <= 512, "two tiles fit");
    // (the boxes are only there where the output leaves through tensor stores: without them a CTA can become resident beside the
    // staging kernel's and overlap its prologue)
    static constexpr int smem_bytes(bool boxes) { return STAGES * STAGE_BYTES + 256 /*barriers*/ + (boxes ? STORE_BYTES : 0) + 1024 /*alignment*/; }
};

// ---- cta_group::2 forms of the wrappers in tc_ptx.cuh.  `bar` of a load is a cluster address (the first CTA's barrier).
__device__ __forceinline__ void load_im2col(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c, int w, int h, int n, uint16_t ow, uint16_t oh)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.im2col.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6}], [%2], {%7, %8};"
        :: "r"(dst), "l"((uint64_t)map), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n), "h"(ow), "h"(oh) : "memory");
}
__device__ __forceinline__ void load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, int z)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        :: "r"(dst), "l"((uint64_t)map), "r"(bar), "r"(x), "r"(y), "r"(z) : "memory");
}
__device__ __forceinline__ void commit_both(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 :: "r"(bar), "h"((uint16_t)3) : "memory");
}
template <bool F16>
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate)
{
    if constexpr (F16)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                     :: "r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
                     :: "r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
// the same operand formats as the one-CTA kernels, M = 256
template <int BN, bool F16>
__host__ __device__ constexpr uint32_t instr_desc()
{
    return ((F16 ? instr_desc_f16<BN>() : instr_desc_tf32<BN>()) & ~(0x1Fu << 24)) | ((uint32_t)(256 >> 4) << 24);
}

template <int BN, bool F16, bool MULTI>
__global__ void __launch_bounds__(kThreads, 1)
pair_conv_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, const __grid_constant__ CUtensorMap map_o,
                 const PairParams p)
{
    using C = Cfg<BN>;
    constexpr int STAGES = C::STAGES, CH = F16 ? 64 : 32;
    constexpr int ACCS = MULTI ? C::ACCS : 1, TILE_COLS = ACCS * BN;
    constexpr int TMEM_COLS = 2 * TILE_COLS <= 128 ? 128 : 2 * TILE_COLS <= 256 ? 256 : 512;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    constexpr int CPS = C::CPS, A_STAGE_BYTES = CPS * A_CHUNK_BYTES, B_STAGE_BYTES = CPS * C::B_CHUNK_BYTES;
    const uint32_t smem_a = smem_base, smem_b = smem_base + STAGES * A_STAGE_BYTES;
    const uint32_t store = smem_base + STAGES * C::STAGE_BYTES;                // 8 boxes, one per epilogue warp
    const uint32_t bars = store + (p.out_tma ? C::STORE_BYTES : 0);
    const uint32_t full_bar = bars, empty_bar = bars + 8 * STAGES;
    const uint32_t acc_full = bars + 16 * STAGES, acc_empty = acc_full + 16;    // two each
    __shared__ uint32_t s_tmem_base;
    __shared__ volatile int s_abort;
    __shared__ __align__(16) float s_bias[2][BN];

    const int warp = uniform_warp_index(), lane = threadIdx.x & 31;
    const uint32_t rank = cluster_cta_rank();
    const int pair_id = (int)blockIdx.x >> 1, pairs = (int)gridDim.x >> 1;

    pdl_launch_dependents();
    if (threadIdx.x == 0) {
        s_abort = 0;
        for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar + 8 * s, 1); mbar_init(empty_bar + 8 * s, 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(acc_full + 8 * s, 1); mbar_init(acc_empty + 8 * s, 16); }      // 8 epilogue warps per CTA
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        prefetch_tensormap(&map_a);
        prefetch_tensormap(&map_b);
        if (p.out_tma) prefetch_tensormap(&map_o);
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem_base)), "r"((uint32_t)TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();              // the peer's barriers exist from here on
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, s_tmem_base, 0);
    if (!(p.b_early && warp >= 11)) pdl_wait();

    if (warp == 0) {
        {
            // ---------------- this CTA's 128 input rows
            uint32_t stage = 0, par = 1;
            const uint32_t full0 = map_to_cta(full_bar, 0);
            bool ok = true;
            for (int t = pair_id; t < p.tiles_total && ok; t += pairs) {
                const int m0 = (t / p.tiles_n) * 256 + (int)rank * 128;
                const int n0 = m0 / p.o.PQ, rem = m0 - n0 * p.o.PQ, p0 = rem / p.o.Q, q0 = rem - p0 * p.o.Q;
                const int w0 = q0 * p.stride - p.pad, h0 = p0 * p.stride - p.pad;
                const int cend = p.cchunks * CH;
                int cx = 0, r = 0, s = 0;
                for (int i = 0; i < p.iters; i += CPS) {
                    ok = warp_wait(empty_bar + 8 * stage, par, &s_abort, p.status, 61);
                    if (!ok) break;
#pragma unroll
                    for (int c = 0; c < CPS; ++c) {
                        if (c > 0 && i + c >= p.iters) break;
                        if (elect_one()) load_im2col(smem_a + stage * A_STAGE_BYTES + c * A_CHUNK_BYTES, &map_a, full0 + 8 * stage, cx, w0, h0, n0, (uint16_t)s, (uint16_t)r);
                        cx += CH;
                        if (cx == cend) { cx = 0; if (++s == p.S) { s = 0; ++r; } }
                    }
                    if (++stage == (uint32_t)STAGES) { stage = 0; par ^= 1u; }
                }
            }
        }
    } else if (warp == 11) {
        {
            // ---------------- this CTA's half of the filter rows
            uint32_t stage = 0, par = 1;
            const uint32_t full0 = map_to_cta(full_bar, 0);
            bool ok = true;
            for (int t = pair_id; t < p.tiles_total && ok; t += pairs) {
                const int k0 = (t % p.tiles_n) * BN + (int)rank * C::B_ROWS;
                const int cend = p.cchunks * CH;
                int cx = 0, tap = 0;
                for (int i = 0; i < p.iters; i += CPS) {
                    ok = warp_wait(empty_bar + 8 * stage, par, &s_abort, p.status, 62);
                    if (!ok) break;
#pragma unroll
                    for (int c = 0; c < CPS; ++c) {
                        if (c > 0 && i + c >= p.iters) break;
                        if (elect_one()) load_3d(smem_b + stage * B_STAGE_BYTES + c * C::B_CHUNK_BYTES, &map_b, full0 + 8 * stage, cx, k0, tap);
                        cx += CH;
                        if (cx == cend) { cx = 0; ++tap; }
                    }
                    if (++stage == (uint32_t)STAGES) { stage = 0; par ^= 1u; }
                }
            }
        }
    } else if (warp == 12) {
        if (rank == 0) {
            // ---------------- byte counts of both CTAs' loads
            uint32_t stage = 0, par = 1;
            constexpr uint32_t CHUNK = 2u * (A_CHUNK_BYTES + C::B_CHUNK_BYTES);
            uint32_t extra = pair_id == 0 ? (uint32_t)p.tx_extra : 0u;
            bool ok = true;
            for (int t = pair_id; t < p.tiles_total && ok; t += pairs) {
                for (int i = 0; i < p.iters; i += CPS) {
                    ok = warp_wait(empty_bar + 8 * stage, par, &s_abort, p.status, 63);
                    if (!ok) break;
                    if (elect_one()) mbar_expect_tx(full_bar + 8 * stage, (i + CPS <= p.iters ? CPS * CHUNK : CHUNK) + extra);
                    extra = 0;
                    if (++stage == (uint32_t)STAGES) { stage = 0; par ^= 1u; }
                }
            }
        }
    } else if (warp == 1) {
        if (rank == 0) {
            // ---------------- MMA issue.  The whole warp walks the loop, so that descriptors and addresses stay warp-uniform; one
            // elected lane issues.  (The vote makes a wait that ran out everyone's: no lane is left alone at the election.)
            constexpr uint32_t idesc = instr_desc<BN, F16>();
            const uint64_t da0 = smem_desc_k_sw128(smem_a), db0 = smem_desc_k_sw128(smem_b);
            uint32_t stage = 0, par = 0;
            const int accs = ACCS > 1 ? p.accs : 1;
            bool ok = true, landed = false;
            int local = 0;
            for (int t = pair_id; t < p.tiles_total && ok; t += pairs, ++local) {
                const uint32_t slot = (uint32_t)local & 1u;
                ok = warp_wait(acc_empty + 8 * slot, ((uint32_t)(local >> 1) & 1u) ^ 1u, &s_abort, p.status, 64);
                if (!ok) break;
                tc_fence_after();
                const uint32_t acc0 = tmem + slot * (uint32_t)TILE_COLS;
                uint32_t acc = acc0;
                int chunk = 0;
                for (int i = 0; i < p.iters; i += CPS) {
                    if (!landed) {
                        ok = warp_wait(full_bar + 8 * stage, par, &s_abort, p.status, 65);
                        if (!ok) break;
                    }
                    tc_fence_after();
                    // the next stage's barrier is tested before this stage's MMAs go out: the test's latency runs under their issue
                    // (a test that never suspends: after the last step nothing will arrive, and the commits below must not wait)
                    const uint32_t next = stage + 1 == (uint32_t)STAGES ? 0 : stage + 1, next_par = next == 0 ? par ^ 1u : par;
                    const bool peek = mbar_test_wait(full_bar + 8 * next, next_par);
                    const uint64_t da = da0 + (uint64_t)(stage * (A_STAGE_BYTES >> 4)), db = db0 + (uint64_t)(stage * (B_STAGE_BYTES >> 4));
                    const bool last0 = ++chunk == p.cchunks;
                    if (last0) chunk = 0;
                    const int ks0 = last0 ? p.last_ksteps : 4;
                    int ks1 = 0;
                    if (CPS == 2 && i + 1 < p.iters) {
                        const bool last1 = ++chunk == p.cchunks;
                        if (last1) chunk = 0;
                        ks1 = last1 ? p.last_ksteps : 4;
                    }
                    const bool used = i >= accs * CPS;                // the accumulator holds an earlier stage's sums
                    if (elect_one()) {
                        if (CPS == 2 && ks0 + ks1 == 8) {
#pragma unroll
                            for (int k = 0; k < 8; ++k)
                                mma<F16>(acc, da + (k >> 2) * (A_CHUNK_BYTES >> 4) + 2 * (k & 3), db + (k >> 2) * (C::B_CHUNK_BYTES >> 4) + 2 * (k & 3),
                                         idesc, (used || k) ? 1u : 0u);
                        } else if (CPS == 1 && ks0 == 4) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) mma<F16>(acc, da + 2 * k, db + 2 * k, idesc, (used || k) ? 1u : 0u);
                        } else {
                            for (int k = 0; k < ks0; ++k) mma<F16>(acc, da + 2 * k, db + 2 * k, idesc, (used || k) ? 1u : 0u);
                            for (int k = 0; k < ks1; ++k)
                                mma<F16>(acc, da + (A_CHUNK_BYTES >> 4) + 2 * k, db + (C::B_CHUNK_BYTES >> 4) + 2 * k, idesc, 1u);
                        }
                        commit_both(empty_bar + 8 * stage);
                        if (i + CPS >= p.iters) commit_both(acc_full + 8 * slot);
                    }
                    if (ACCS > 1) { acc += (uint32_t)BN; if (acc == acc0 + (uint32_t)(accs * BN)) acc = acc0; }
                    landed = __all_sync(0xffffffffu, peek);
                    stage = next;
                    par = next_par;
                }
            }
        }
    } else if (warp != 6) {
        // ---------------- epilogue: warps 2..5 take the first half of the channels, 7..10 the second
        const int quarter = warp & 3, group = warp >= 7 ? 1 : 0;
        const int etid = threadIdx.x - (group ? 96 : 64);
        constexpr int NCH = BN / 32, HALF = (NCH + 1) / 2;
        static_assert(NCH >= 2, "both groups have channels, and with them a last chunk that hands the accumulator back");
        const int c_begin = group ? HALF : 0, c_end = group ? NCH : HALF;
        const uint32_t box = store + (uint32_t)(4 * group + quarter) * BOX_BYTES;
        const uint32_t empty0 = map_to_cta(acc_empty, 0);
        const int accs = ACCS > 1 ? p.accs : 1;
        int local = 0;
        for (int t = pair_id; t < p.tiles_total; t += pairs, ++local) {
            const int tm = t / p.tiles_n, k0 = (t - tm * p.tiles_n) * BN;
            const int row0 = tm * 256 + (int)rank * 128 + 32 * quarter, m = row0 + lane;
            const uint32_t slot = (uint32_t)local & 1u;
            float* bias = s_bias[slot];                // its readers of two tiles ago are past the barrier of the tile in between
            for (int j = etid; j < BN; j += 256) bias[j] = (p.bias && k0 + j < p.o.K) ? __ldg(p.bias + k0 + j) : 0.f;
            RowDst d;
            {
                const bool valid = m < p.M;
                const int n = valid ? m / p.o.PQ : 0, pq = valid ? m - n * p.o.PQ : 0, pp = pq / p.o.Q;
                d = row_dst(p.o, valid, n, pp, pq - pp * p.o.Q);
            }
            if (lane == 0) (void)mbar_wait_relaxed(acc_full + 8 * slot, (uint32_t)(local >> 1) & 1u, &s_abort, p.status, 66);
            __syncwarp();
            uint32_t stop;
            asm volatile("{\n\t.reg .pred q, r;\n\tsetp.ne.u32 q, %1, 0;\n\tbar.red.or.pred r, 1, 256, q;\n\tselp.u32 %0, 1, 0, r;\n\t}"
                         : "=r"(stop) : "r"((uint32_t)s_abort) : "memory");
            if (stop) break;
            tc_fence_after();
            const uint32_t trow = tmem + ((uint32_t)(quarter * 32) << 16) + slot * (uint32_t)TILE_COLS;
#pragma unroll 1
            for (int c = c_begin; c < c_end; ++c) {
                uint32_t v[32];
                tmem_ld_32cols(trow + 32 * c, v);
                tmem_ld_wait();
#pragma unroll 1
                for (int a = 1; a < accs; ++a) {
                    uint32_t u[32];
                    tmem_ld_32cols(trow + (uint32_t)(a * BN + 32 * c), u);
                    tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) + __uint_as_float(u[j]));
                }
                if (c + 1 == c_end) {                  // the accumulator has been read: hand it back to the issuer
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" :: "r"(empty0 + 8 * slot) : "memory");
                }
                float y[32];
                bias_relu32(v, bias + 32 * c, p.o.relu != 0, y);
                if (p.out_tma) {
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");      // the box has left
                    __syncwarp();
                    const uint32_t a = box + 128u * (uint32_t)lane;
#pragma unroll
                    for (int g = 0; g < 8; ++g)
                        st_shared_v4(a + (uint32_t)((g ^ (lane & 7)) << 4), round_to_tf32(y[4 * g]), round_to_tf32(y[4 * g + 1]),
                                     round_to_tf32(y[4 * g + 2]), round_to_tf32(y[4 * g + 3]));
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0 && k0 + 32 * c < p.o.Cp && row0 < p.M) {
                        tma_store_2d(&map_o, box, k0 + 32 * c, row0);
                        bulk_commit();
                    }
                } else {
                    store_row32(p.o, d, k0 + 32 * c, y);
                }
            }
        }
        if (p.out_tma && lane == 0) bulk_wait_all();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();              // nobody leaves while the peer may still signal its barriers or its MMAs read this shared memory
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)TMEM_COLS) : "memory");
    }
}

}  // namespace pair
}  // namespace boda
