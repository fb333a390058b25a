// TCONV for stride-1 layers straight from the NCHW input: nothing is staged in global memory.
//
// The window reuse is the halo kernel's (tconv_halo.cuh): output positions are numbered through an image padded on the right and
// below, f = (n*Hp + p)*Wp + q with Hp = H + pad and Wp = W + pad, so that under tap (r, s) position f reads slab row f - f0 + r*Wp + s,
// and a tap is one A descriptor that starts that many 128-byte rows into the slab.  Here the slab is built by eight warps from the tensor as it
// lies: a lane takes a position, a warp 16 bytes of its row (four channels of fp32, eight of fp16), so that loads run along image
// rows, the swizzled 16-byte stores meet no bank twice, and rounding costs nothing extra.
// What that is for:
//  * The staging launch in front of the im2col, halo and pair kernels, with its pass over the input, was 4 to 6 us of a layer.
//  * The im2col kernels fetch every input row once per tap, and L2 gives them some 16 KB a clock in all (fitted, see model_cost).  A slab is filled once per
//    chunk of channels, and what is left are the filters: BN rows a tap where they fetch 128 + BN.  Narrow tiles then cost little, so that a
//    round of 148 CTAs fills without a split of the reduction over a cluster and its exchange.
// The price: positions right of and below the image are computed and dropped (7 to 16 % of the rows for 13x13 and 27x27).
// Measured, a call of a plan with its output allocated: 3x3 on 256 channels, 384 filters, 13x13, batch 20 19.1 us (im2col 128x192, split) -> 15.7 (128x96); 5x5 on
// 96 channels, 256 filters, 27x27, batch 20 with fp16 operands 25.1 (pairs) -> 23.0 (128x256).
//
// The tile's width BN is a run-time value (a multiple of 16), chosen so that the tiles fill whole rounds of the SMs.  MMAs of 128 x BN x 32
// bytes take max(BN/2, 32 + BN/4) clocks: below 128 channels the tensor core waits for its operands from shared memory.  A stage of
// filters holds TPS taps of a window row, so that the issuing warps' waits, votes and commits are few beside a narrow tile's MMAs.  A chunk costs
// some 500 clocks besides its stages, a further tile of a CTA 6000, in which the second set of builders stores instead of building: layers of
// several rounds are mostly left to the pairs.  Two sets of builders beside eight warps for the epilogue (896 threads, 72 registers)
// were slower than sharing them (conv3 at batch 20: 20.8 us, 16.1).
//
// Roles (640 threads): warps 0 and 2 = filters by TMA, warps 1 and 3 = MMA issue (warp 1 also tensor memory), warps 4..19 = slab builders, of which
// warps 4..11 store the tiles.  Persistent.  With a
// split, CTA z of a cluster takes chunks [z*chunks_per_split, ...), parks its sums in shared memory and adds its share of the
// channels in rank order.  All waits are bounded as elsewhere.
#pragma once

#include "tc_ptx.cuh"
#include "pair_conv.cuh"

#include <cuda_fp16.h>

#include <type_traits>

namespace boda {
namespace slab {

using namespace tc;

constexpr int kFirstEpilogueWarp = 4, kFirstBuilderWarp = 12;
constexpr int kThreads = 32 * (kFirstBuilderWarp + 8);       // 640
constexpr int kSlots = 2;                                    // slabs
constexpr int kMaxStages = 8;
constexpr int kMaxGroups = 16;                               // a slab is at most 512 rows
constexpr int kMaxBN = 256;
constexpr int kBarrierBytes = 512;
constexpr int kSmemBudget = 222 * 1024;

// Division of numbers below 2^31 (Granlund and Montgomery, Division by Invariant Integers using Multiplication, 1994): multiply by ceil(2^(31 + l) / d),
// l = ceil(log2 d), and shift.
struct FastDiv {
    unsigned mul, shift;
    static FastDiv of(unsigned d)
    {
        unsigned l = 0;
        while ((1ull << l) < d) ++l;
        return {d == 1 ? 0u : (unsigned)(((1ull << (31 + l)) + d - 1) / d), d == 1 ? 0u : l - 1};
    }
    __device__ __forceinline__ int div(int x) const { return mul ? (int)(__umulhi((unsigned)x, mul) >> shift) : x; }
};

struct SlabParams {
    const float* in;
    int C, H, W, HW;
    unsigned CHW;
    int Mflat, HpWp, Wp;         // flat positions
    FastDiv by_image, by_row;    // by HpWp and Wp
    int lead;                    // pad*Wp + pad: slab row 0 is the input of position f0 - lead
    int S, taps;
    int cchunks;                 // chunks of 128 bytes of channels
    int last_ksteps;             // MMA steps of the last chunk that hold channels
    int slab_rows, slab_bytes;
    int BN, b_stages, b_tap_bytes, b_stage_bytes;
    int accs;                    // accumulators of a tile, one per issuing warp (1 or 2)
    int slots;                   // tiles under way (1 or 2)
    int tmem_cols;
    uint32_t idesc;
    int splits, chunks_per_split;
    int tiles_n, tiles_total;    // tiles are numbered position tile * tiles_n + channel tile
    const float* bias;
    OutSpec o;                   // NCHW
    int* status;
    int tx_extra;                // test hook: bytes added to the expected size of the first stage of the first CTA
    int b_early;                 // bound filters: their loads need not wait for the preceding kernel
};

__device__ __forceinline__ void tmem_ld_16cols(uint32_t taddr, uint32_t (&v)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ uint32_t half_pair(float a, float b)
{
    const __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// element offset of flat input position f inside channel 0 of its image; -1: padding, reads as zeros
__device__ __forceinline__ int position_offset(const SlabParams& p, int f)
{
    if (f < 0 || f >= p.Mflat) return -1;
    const int n = p.by_image.div(f), rem = f - n * p.HpWp, y = p.by_row.div(rem), x = rem - y * p.Wp;
    return y < p.H && x < p.W ? (int)((unsigned)n * p.CHW) + y * p.W + x : -1;
}
// image and output point of flat position f; not valid right of and below the output
struct OutPos { bool valid; int n, pq; };
__device__ __forceinline__ OutPos out_position(const SlabParams& p, int f)
{
    OutPos d = {f < p.Mflat, 0, 0};
    if (d.valid) {
        d.n = p.by_image.div(f);
        const int rem = f - d.n * p.HpWp, pp = p.by_row.div(rem), qq = rem - pp * p.Wp;
        d.valid = pp < p.o.P && qq < p.o.Q;
        d.pq = d.valid ? pp * p.o.Q + qq : 0;
    }
    return d;
}

// Split reduction: every CTA of the cluster has parked its sums at smem_base, [channel][128 rows]; each adds its share of the channels over
// all of them in rank order.  Called by all threads; `row` and `group` are those of the epilogue warps.
__device__ __forceinline__ void cluster_add_store(const SlabParams& p, int BN, uint32_t smem_base, int warp, int row, int group, int aborted)
{
    cluster_sync_all();
    if (warp >= kFirstEpilogueWarp && warp < kFirstBuilderWarp && aborted == 0) {
        const int rank = (int)cluster_cta_rank(), tm = (int)blockIdx.x / p.tiles_n, k0 = ((int)blockIdx.x - tm * p.tiles_n) * BN;
        const OutPos d = out_position(p, tm * 128 + row);
        float* out = p.o.out + ((size_t)d.n * p.o.K + k0) * p.o.PQ + d.pq;
        const int share_end = (rank + 1) * BN / p.splits;
        uint32_t peer[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) peer[r] = map_to_cta(smem_base + (uint32_t)row * 4u, (uint32_t)min(r, p.splits - 1));
        // four channels at a time, all the peers' values of them in flight before the first is added
        for (int c = rank * BN / p.splits + group; c < share_end; c += 8) {
            float x[8][4];
#pragma unroll
            for (int r = 0; r < 8; ++r)
#pragma unroll
                for (int u = 0; u < 4; ++u) x[r][u] = r < p.splits && c + 2 * u < share_end ? ld_cluster_f32(peer[r] + (uint32_t)(c + 2 * u) * 512u) : 0.f;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = c + 2 * u;
                if (k >= share_end || k0 + k >= p.o.K) break;
                float y = x[0][u];
#pragma unroll
                for (int r = 1; r < 8; ++r)
                    if (r < p.splits) y += x[r][u];
                if (p.bias) y += __ldg(p.bias + k0 + k);
                if (p.o.relu) y = fmaxf(y, 0.f);
                if (d.valid) out[(size_t)k * p.o.PQ] = y;
            }
        }
    }
    cluster_sync_all();          // nobody leaves while a peer may still read its shared memory
}

template <bool F16, int TPS>
__global__ void __launch_bounds__(kThreads, 1)
slab_conv_kernel(const __grid_constant__ CUtensorMap map_b, const SlabParams p)
{
    constexpr int CH = F16 ? 64 : 32;            // channels per chunk: 128 bytes
    constexpr int VPT = F16 ? 8 : 4;             // channels that a builder thread loads: 16 bytes
    constexpr int BATCH = 32 / VPT;              // positions of a thread whose loads are in flight together
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t smem_b = smem_base + (uint32_t)(kSlots * p.slab_bytes);
    const uint32_t bars = smem_b + (uint32_t)(p.b_stages * p.b_stage_bytes);
    const uint32_t b_full = bars, b_empty = b_full + 8 * kMaxStages;
    const uint32_t a_full = b_empty + 8 * kMaxStages, a_empty = a_full + 8 * kSlots;
    const uint32_t acc_full = a_empty + 8 * kSlots, acc_empty = acc_full + 16;
    __shared__ uint32_t s_tmem_base;
    __shared__ volatile int s_abort;
    __shared__ __align__(16) float s_bias[2][kMaxBN];

    const int warp = uniform_warp_index(), lane = threadIdx.x & 31;
    const int c_begin = (int)blockIdx.z * p.chunks_per_split, c_end = min(p.cchunks, c_begin + p.chunks_per_split);

    pdl_launch_dependents();
    if (threadIdx.x == 0) {
        s_abort = 0;
        for (int s = 0; s < p.b_stages; ++s) { mbar_init(b_full + 8 * s, 1); mbar_init(b_empty + 8 * s, 1); }
        for (int s = 0; s < kSlots; ++s) { mbar_init(a_full + 8 * s, 8); mbar_init(a_empty + 8 * s, p.accs); }  // 8 warps build a slab
        for (int s = 0; s < 2; ++s) { mbar_init(acc_full + 8 * s, p.accs); mbar_init(acc_empty + 8 * s, 8); }   // 8 epilogue warps
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        prefetch_tensormap(&map_b);
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&s_tmem_base), (uint32_t)p.tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, s_tmem_base, 0);
    if (warp < kFirstEpilogueWarp && !(p.b_early && (warp == 0 || warp == 2))) pdl_wait();       // the others compute positions first

    const int quarter = warp & 3, group = warp >= kFirstEpilogueWarp + 4 ? 1 : 0, row = 32 * quarter + lane;      // epilogue warps

    if (warp == 0 || warp == 2) {
        // ---------------- filters: TPS taps of a window row per stage, one box; warp 0 fills the even stages of the ring, warp 2 the odd ones.  (Whole
        // warps walk the loop and an elected lane issues: the same in a branch of one lane, whose addresses are not warp-uniform, takes several
        // times as long.)
        const uint32_t me = warp == 0 ? 0u : 1u, stage_bytes = (uint32_t)p.b_stage_bytes;
        const uint32_t full0 = b_full + 8 * me, empty0 = b_empty + 8 * me, dst0 = smem_b + me * stage_bytes, full_end = full0 + 8 * (uint32_t)p.b_stages;
        uint32_t fb = full0, eb = empty0, par = 1, dst = dst0;
        uint32_t extra = (blockIdx.x | blockIdx.z | me) == 0 ? (uint32_t)p.tx_extra : 0u;
        const int taps = p.taps, c_last = c_end * CH;
        bool ok = true;
        int tap = (int)me * TPS;
        for (int t = blockIdx.x; t < p.tiles_total && ok; t += gridDim.x) {
            const int k0 = (t % p.tiles_n) * p.BN;
            for (int cx = c_begin * CH; cx < c_last && ok; cx += CH, tap -= taps) {
                for (; tap < taps; tap += 2 * TPS) {
                    ok = warp_wait(eb, par, &s_abort, p.status, 82);
                    if (!ok) break;
                    if (elect_one()) {
                        mbar_expect_tx(fb, stage_bytes + extra);
                        tma_load_3d(dst, &map_b, fb, cx, k0, tap);
                    }
                    __syncwarp();
                    extra = 0;
                    fb += 16; eb += 16; dst += 2 * stage_bytes;
                    if (fb == full_end) { fb = full0; eb = empty0; dst = dst0; par ^= 1u; }
                }
            }
        }
    } else if (warp == 1 || (warp == 3 && p.accs > 1)) {
        // ---------------- MMA issue: the whole warp walks the loop (descriptors stay warp-uniform), one elected lane issues.  A commit holds its
        // thread for 150 clocks and the rest of a stage's bookkeeping for some 200, while the tensor core's queue covers three or four
        // MMAs: two warps take the stages in turn (the ring has an even number of them), each into its own accumulator.
        // Literal offsets inside a stage, descriptors and barriers advanced by additions.
        const uint32_t me = warp == 1 ? 0u : 1u, accs = (uint32_t)p.accs;
        const uint64_t da0 = smem_desc_k_sw128(smem_base), db0 = smem_desc_k_sw128(smem_b) + me * (uint32_t)(p.b_stage_bytes >> 4);
        const uint64_t pitch = 8ull * (uint64_t)p.Wp, slab_step = (uint64_t)(p.slab_bytes >> 4);              // a window row; 16-byte units
        const uint32_t tap_step = (uint32_t)p.b_tap_bytes >> 4, stage_step = accs * ((uint32_t)p.b_stage_bytes >> 4);
        const uint32_t idesc = p.idesc, full0 = b_full + 8 * me, empty0 = b_empty + 8 * me, full_end = full0 + 8 * (uint32_t)p.b_stages, ring = 8 * accs;
        const int per_row = p.S / TPS, groups = p.taps / TPS;
        const uint64_t row_step = pitch - 8 * TPS * (uint32_t)per_row;      // from behind a window row's last tap to the next row's first
        uint32_t fb = full0, eb = empty0, par = 0, aslot = 0, apar = 0;
        uint64_t db = db0;
        bool ok = true;
        int local = 0, g = (int)me;                          // this warp's next stage within the chunk
        for (int t = blockIdx.x; t < p.tiles_total && ok; t += gridDim.x, ++local) {
            const uint32_t slot = p.slots > 1 ? (uint32_t)local & 1u : 0u, use = (uint32_t)(p.slots > 1 ? local >> 1 : local);
            ok = warp_wait(acc_empty + 8 * slot, (use & 1u) ^ 1u, &s_abort, p.status, 84);
            if (!ok) break;
            tc_fence_after();
            const uint32_t acc = tmem + (slot * accs + me) * (uint32_t)p.BN;
            uint32_t goes_on = 0;
            for (int c = c_begin; c < c_end; ++c) {
                ok = warp_wait(a_full + 8 * aslot, apar, &s_abort, p.status, 83);
                if (!ok) break;
                const int ksteps = c + 1 == p.cchunks ? p.last_ksteps : 4;
                const uint64_t slab = da0 + (aslot ? slab_step : 0);
                auto chunk = [&](auto all_steps) {
                    int s = per_row > 1 ? g : 0;             // g is 0 or 1 here
                    uint64_t da = slab + (g == 0 ? 0 : per_row > 1 ? 8 * TPS : pitch);
                    for (; g < groups; g += (int)accs) {
                        ok = warp_wait(fb, par, &s_abort, p.status, 85);
                        if (!ok) return;
                        tc_fence_after();
                        if (elect_one()) {
#pragma unroll
                            for (int i = 0; i < TPS; ++i)
#pragma unroll
                                for (int k = 0; k < 4; ++k)
                                    if (decltype(all_steps)::value || k < ksteps) {
                                        if constexpr (F16) umma_f16(acc, da + 8 * i + 2 * k, db + i * tap_step + 2 * k, idesc, i | k ? 1u : goes_on);
                                        else umma_tf32(acc, da + 8 * i + 2 * k, db + i * tap_step + 2 * k, idesc, i | k ? 1u : goes_on);
                                    }
                            tc_commit(eb);
                        }
                        __syncwarp();
                        goes_on = 1u;
                        fb += ring; eb += ring; db += stage_step;
                        if (fb == full_end) { fb = full0; eb = empty0; db = db0; par ^= 1u; }
                        s += (int)accs;
                        da += 8 * TPS * accs;
                        if (s >= per_row) { s -= per_row; da += row_step; }
                        if (s >= per_row) { s -= per_row; da += row_step; }
                    }
                };
                if (ksteps == 4) chunk(std::true_type());
                else chunk(std::false_type());
                if (!ok) break;
                g -= groups;
                if (elect_one()) {
                    tc_commit(a_empty + 8 * aslot);
                    if (c + 1 == c_end) tc_commit(acc_full + 8 * slot);
                }
                __syncwarp();
                aslot ^= 1u;
                if (aslot == 0) apar ^= 1u;
            }
        }
    } else if (warp >= kFirstEpilogueWarp) {
        // ---------------- slab builders: two sets of eight warps, one for each slab (a chunk's loads, conversions and stores are a chain of some 2000
        // clocks, as long as the MMAs of a whole chunk of a 3x3 layer).  Warp `piece` of a set fills 16-byte piece `piece` of every row, lanes along
        // the positions.  The second set (warps 4..11) stores the tile as well.
        const int piece = (warp - kFirstEpilogueWarp) & 7, set = warp >= kFirstBuilderWarp ? 0 : 1;
        const int ngroups = (p.slab_rows + 31) >> 5;
        const uint32_t dst = smem_base + (uint32_t)(set * p.slab_bytes) + (uint32_t)lane * 128u + (uint32_t)((piece ^ (lane & 7)) << 4);
        const uint32_t empty = a_empty + 8 * (uint32_t)set, full = a_full + 8 * (uint32_t)set;
        const int etid = threadIdx.x - 32 * kFirstEpilogueWarp, pieces = p.BN / 16;
        uint32_t par = 1;
        bool ok = true;
        int c = c_begin + set, local = 0;                                        // c: this set's next chunk
        for (int t = blockIdx.x; t < p.tiles_total; t += gridDim.x, ++local) {
            const int tm = t / p.tiles_n;
            {
                const int f_first = tm * 128 - p.lead + lane;
                int off[kMaxGroups];
#pragma unroll
                for (int g = 0; g < kMaxGroups; ++g) off[g] = g < ngroups ? position_offset(p, f_first + 32 * g) : -1;
                if (local == 0) pdl_wait();
                for (; c < c_end; c += 2) {
                    if (!ok) continue;
                    const int ch = c * CH + piece * VPT, live = p.C - ch;        // channels from ch on that exist
                    const float* base = p.in + (size_t)ch * p.HW;
#pragma unroll
                    for (int b = 0; b < kMaxGroups / BATCH; ++b) {
                        if (b * BATCH >= ngroups) break;
                        float v[BATCH][VPT];
#pragma unroll
                        for (int g = 0; g < BATCH; ++g)
                            if (b * BATCH + g < ngroups) {
#pragma unroll
                                for (int u = 0; u < VPT; ++u)
                                    v[g][u] = off[b * BATCH + g] >= 0 && u < live ? __ldg(base + (size_t)u * p.HW + off[b * BATCH + g]) : 0.f;
                            }
                        if (b == 0) {
                            // the loads are in flight while this waits for the slab to be free (one poller per warp, a warp-wide decision)
                            int free_now = 0;
                            if (lane == 0) free_now = mbar_test_wait(empty, par) || mbar_wait_relaxed(empty, par, &s_abort, p.status, 81) ? 1 : 0;
                            ok = __shfl_sync(0xffffffffu, free_now, 0) != 0;
                            if (!ok) break;
                            __syncwarp();
                            par ^= 1u;
                        }
#pragma unroll
                        for (int g = 0; g < BATCH; ++g) {
                            const int r = 32 * (b * BATCH + g);
                            if (r + lane < p.slab_rows) {
                                const uint32_t a = dst + (uint32_t)r * 128u;
                                if constexpr (F16)
                                    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" :: "r"(a), "r"(half_pair(v[g][0], v[g][1])),
                                                 "r"(half_pair(v[g][2], v[g][3])), "r"(half_pair(v[g][4], v[g][5])), "r"(half_pair(v[g][6], v[g][7])) : "memory");
                                else
                                    st_shared_v4(a, round_to_tf32(v[g][0]), round_to_tf32(v[g][1]), round_to_tf32(v[g][2]), round_to_tf32(v[g][3]));
                            }
                        }
                    }
                    if (!ok) continue;
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(full) : "memory");
                }
                c -= c_end - c_begin;
            }
            if (set == 0) {
                if (!ok) break;
                continue;
            }
            // ---------------- epilogue: warps 4..7 take the even 16-channel pieces of the accumulator, warps 8..11 the odd ones.  (A warp whose wait ran
            // out above comes here too: the barrier below takes the common decision.)
            const int k0 = (t - tm * p.tiles_n) * p.BN;
            const uint32_t slot = p.slots > 1 ? (uint32_t)local & 1u : 0u, use = (uint32_t)(p.slots > 1 ? local >> 1 : local);
            float* bias = s_bias[local & 1];           // its readers of two tiles ago are past the barrier of the tile in between
            for (int j = etid; j < p.BN; j += 256) bias[j] = (p.bias && k0 + j < p.o.K) ? __ldg(p.bias + k0 + j) : 0.f;
            const OutPos d = out_position(p, tm * 128 + row);
            float* out = p.o.out + ((size_t)d.n * p.o.K + k0) * p.o.PQ + d.pq;
            if (lane == 0) (void)mbar_wait_relaxed(acc_full + 8 * slot, use & 1u, &s_abort, p.status, 86);
            __syncwarp();
            uint32_t stop;
            asm volatile("{\n\t.reg .pred q, r;\n\tsetp.ne.u32 q, %1, 0;\n\tbar.red.or.pred r, 1, 256, q;\n\tselp.u32 %0, 1, 0, r;\n\t}"
                         : "=r"(stop) : "r"((uint32_t)s_abort) : "memory");
            if (stop) break;
            tc_fence_after();
            const uint32_t trow = tmem + ((uint32_t)(32 * quarter) << 16) + slot * (uint32_t)(p.accs * p.BN);
#pragma unroll 1
            for (int e = group; e < pieces; e += 2) {
                uint32_t v[16], u[16];
                tmem_ld_16cols(trow + 16 * e, v);
                if (p.accs > 1) tmem_ld_16cols(trow + (uint32_t)(p.BN + 16 * e), u);
                tmem_ld_wait();
                if (p.accs > 1) {
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) + __uint_as_float(u[j]));
                }
                if (p.splits > 1) {
                    // this CTA's sums, [channel][128 rows], for the peers (the stages are idle: a CTA of a split has one tile)
#pragma unroll
                    for (int j = 0; j < 16; ++j) st_shared_f32(smem_base + (uint32_t)(((16 * e + j) * 128 + row) * 4), __uint_as_float(v[j]));
                    continue;
                }
                float* dst = out + (size_t)(16 * e) * p.o.PQ;
                const int live = d.valid ? p.o.K - k0 - 16 * e : 0;
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    const float4 b4 = *reinterpret_cast<const float4*>(bias + 16 * e + 4 * g);
                    const float bb[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        float y = __uint_as_float(v[4 * g + j]) + bb[j];
                        if (p.o.relu) y = fmaxf(y, 0.f);
                        if (4 * g + j < live) dst[(size_t)(4 * g + j) * p.o.PQ] = y;
                    }
                }
            }
            if (p.splits > 1) break;
            // the accumulator has been read: hand it back to the issuer
            tc_fence_before();
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(acc_empty + 8 * slot) : "memory");
        }
    }
    if (p.splits > 1) cluster_add_store(p, p.BN, smem_base, warp, row, group, s_abort);
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, (uint32_t)p.tmem_cols);
    }
}

}  // namespace slab
}  // namespace boda
