// Tensor-core MXInt product with the packed weights decoded into TENSOR MEMORY, on CTA pairs.  Sec. 3.2 operator on exactly
// decoded operands, as mx_gemm_tc.cuh, computed transposed: the weights are the A operand of the MMA (a lane of tensor memory
// is an output feature), the activations are B, and the accumulator holds the result with tokens along its columns.
//
// Why: a pass that writes the weights out in bf16 costs four times their packed size in traffic before the product can start,
// and the product on two shared-memory operands is bound by shared memory (mx_gemm_tc2.cuh: 156 bytes per clock wanted, 128
// there; gemm_dec_kernel with three panels as well).  A operands may come from tensor memory, where the decoding warps put them
// with one instruction and without the proxy fence that publishes shared memory; per K step of 64 a CTA then fetches its T / 2
// rows of activations and 4 (8) KB of packed weights, and shared memory serves 64 T bytes written, 128 T read and twice the packed
// ones for 2 T clocks of MMA.
//   warp 0       : activations by TMA, two K steps per stage
//   warp 1       : tensor-memory allocation, MMA issue (the leader's)
//   warp 2       : packed weights: 128 rows x 128 bytes by TMA, exponent bytes by background copies
//   warps 4..15  : three groups that decode every third K step each into one of four or eight stages of 32 columns
//   warps 16..23 : epilogue
// The tile is 256 features x T tokens, T a multiple of 32 that the host picks so that the tiles fill whole rounds of the chip's
// pairs; up to T = 192 there are two accumulators, so the epilogue of a tile runs under the next one's MMAs.  Few tiles: K is cut
// over the pairs of a cluster, whose partial tiles go to shared memory and are added up in the order of K (mx_gemm_splitk.cuh).
// Bound by the instructions of the decoding warps, 0.25 us per K step and round up to T = 160 and 0.26 at 192 (without the MMAs the
// same, without the decoding 0.16 at T = 64 and 0.31 at 256; four groups of warps, two steps per turn of a group, or half of the shifts
// as multiplications changed nothing), and above by the MMAs (T = 224: 453 clocks per step by the counters, of which its MMAs need
// 2 T = 448; 0.30 us at 256).
// Whole calls, M x K x N, against a pass and a product / gemm_dec_kernel: 512 x 4096 x 11008 55.0 -> 45.6 us (with an MXInt result 53.3),
// 256 x 4096 x 12288 42.5 -> 30.5, 128 x 4096 x 11008 30.0 -> 25.0, 352 x 2048 x 6144 19.2 -> 17.0; where it is chosen: tmw_tokens.
// Persistent; all waits are bounded.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "mx_gemm_tc.cuh"
#include "mx_gemv_mma.cuh"
#include "mx_ptx.cuh"
#include "mx_step_walk.h"

namespace mx {

struct TmwCfg {
    static constexpr int BN = 128;                                       // features per CTA
    static constexpr int GROUPS = 3, EPI_WARPS = 8;
    static constexpr int THREADS = 32 * (4 + 4 * GROUPS + EPI_WARPS);
    static constexpr int RAW_STAGES = 4, MAX_A_STAGES = 8, MAX_STAGES = 8;  // of packed weights, decoded weights, activations
    static constexpr uint32_t RAW_MANT = BN * 128, RAW_EXP = BN * 20;    // 128 mantissa bytes and the words of at most 16 exponent bytes per row
    static constexpr uint32_t RAW_BYTES = RAW_STAGES * (RAW_MANT + RAW_EXP);
    static constexpr int MAX_T = 256, MAX_SPLIT = 4;
    // Tensor memory: one accumulator of T columns, or two up to T = 192; behind them the stages of decoded weights, 32 columns each
    static constexpr uint32_t TMEM_COLS = 512;
    static __host__ __device__ constexpr int accs(int T) { return T <= 192 ? 2 : 1; }
    static __host__ __device__ constexpr uint32_t acc_col(int T) { return T <= 128 ? 128 : 192; }
    static __host__ __device__ constexpr uint32_t a_col(int T) { return T <= 128 || T > 192 ? 256 : 384; }
    static __host__ __device__ constexpr int a_stages(int T) { return T <= 128 || T > 192 ? 8 : 4; }
    // A stage of activations holds two K steps: with one, the loop that issues the MMAs took 450 clocks per step, whatever T
    static constexpr uint32_t half_bytes(int T) { return (uint32_t)T * (TC_BK * 2) / 2; }
    static constexpr uint32_t stage_bytes(int T) { return 2 * half_bytes(T); }
    static constexpr uint32_t fixed_bytes(bool qout) { return RAW_BYTES + (qout ? EPI_WARPS * 4096 : 0) + 512 + 1024; }    // qout: transposing buffers
    static constexpr int stages(int T, bool qout)
    {
        const int n = (int)((227 * 1024 - fixed_bytes(qout)) / stage_bytes(T));
        return n < MAX_STAGES ? n : MAX_STAGES;
    }
    static constexpr uint32_t smem_bytes(int T, bool qout) { return stages(T, qout) * stage_bytes(T) + fixed_bytes(qout); }
};

struct TmwParams {
    const uint8_t *w_exp;
    int w_bits, w_rows2, block;
    int tokens;               // T
    int stages;
    int early;                // 1: the launch in front is this call's activation pass
    int exp_words;            // 1: every row's exponent bytes start at a whole word
    int split;                // > 1: pieces of K; a cluster of as many pairs shares one tile, and the grid has a cluster per tile
};

// The exponent bytes of 128 rows of packed weights, for the warp that feeds the decoding ones: a lane owns rows lane, lane + 32,
// ..., whose addresses it works out once per tile, and copies a row's `bytes` per raw stage in the background, in pieces as wide
// as all their addresses are aligned to; where those are no whole words, by the aligned words that hold them.  Bytes behind a
// row's end are zeros.
struct ExpFeed {
    const uint8_t *row[4];
    int nb, bytes, words;     // exponent bytes of a row, per raw stage, and the words that hold the latter
    int unit;                 // 16, 8, 4: every piece is as wide and aligned; 0: by words

    // every stage starts a multiple of `bytes` into the rows (pieces of K are whole raw stages)
    __device__ __forceinline__ ExpFeed(const uint8_t *w_exp, int nb_, int bytes_, int exp_words)
        : nb(nb_), bytes(bytes_), words((bytes_ >> 2) + (exp_words ? 0 : 1))
    {
        const uint32_t all = (uint32_t)reinterpret_cast<uintptr_t>(w_exp) | (uint32_t)nb_ | (uint32_t)bytes_;
        unit = !exp_words ? 0 : (all & 15u) == 0 ? 16 : (all & 7u) == 0 ? 8 : 4;
    }
    __device__ __forceinline__ void rows(const uint8_t *w_exp, int n0, int N, int shift, int lane)
    {
#pragma unroll
        for (int i = 0; i < 4; ++i) row[i] = w_exp + (int64_t)(min(n0 + lane + 32 * i, N - 1) >> shift) * nb;
    }
    // bytes b0 .. of every row (b0 < nb) -> `dst`, 4 * words bytes per row
    __device__ __forceinline__ void copy(uint32_t dst, int b0, int lane) const
    {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t d = dst + (uint32_t)(lane + 32 * i) * 4u * words;
            if (unit == 16) {
                cp_async16(d, row[i] + b0);                              // bytes = 16
            } else if (unit == 8) {
                cp_async8(d, row[i] + b0, 8);
                if (bytes == 16) cp_async8(d + 8, row[i] + (b0 + 8 < nb ? b0 + 8 : 0), b0 + 8 < nb ? 8 : 0);
            } else {
                const int skip = unit ? 0 : (int)((uint32_t)reinterpret_cast<uintptr_t>(row[i]) & 3u);
                for (int w = 0; w < words; ++w) {
                    const int at = b0 + 4 * w - skip, valid = min(nb - at, 4);
                    cp_async4(d + 4 * w, row[i] + (valid > 0 ? at : -skip), max(valid, 0));
                }
            }
        }
    }
};

// 32 tokens from m0 on of feature n (a lane each), r[j] = token m0 + j: bias, ReLU and residual.
__device__ __forceinline__ void tmw_tail(const TcParams &p, int m0, int n, float bias, uint32_t (&r)[32])
{
    const bool live = n < p.N;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        float v = __uint_as_float(r[j]) + bias;
        if (p.relu) v = v < 0.f ? 0.f : v;                               // NaN stays NaN
        r[j] = __float_as_uint(v);
    }
    if (p.residual) {
        const float *src = p.residual + (int64_t)m0 * p.ldr + n;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float x[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) x[j] = live && m0 + 16 * h + j < p.M ? __ldg(src + (int64_t)(16 * h + j) * p.ldr) : 0.f;
#pragma unroll
            for (int j = 0; j < 16; ++j) r[16 * h + j] = __float_as_uint(__uint_as_float(r[16 * h + j]) + x[j]);
        }
    }
}

// A warp's 32 features x 32 tokens, a feature per lane -> a token per lane, r[f] = feature f, through 4 KB of shared memory at
// `buf` (groups of four words swizzled by the token: no bank conflicts on either side).  The MXInt result has its blocks along the
// features; across the lanes each value's block maximum took five shuffles (2048 x 4096 x 16384 476 us against 219 in fp32).
__device__ __forceinline__ void tmw_transpose(uint8_t *buf, int lane, uint32_t (&r)[32])
{
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 32; ++j)
        *reinterpret_cast<uint32_t *>(buf + j * 128 + (((lane >> 2) ^ (j & 7)) << 4) + (lane & 3) * 4) = r[j];
    __syncwarp();
#pragma unroll
    for (int v = 0; v < 8; ++v) {
        const uint4 x = *reinterpret_cast<const uint4 *>(buf + lane * 128 + ((v ^ (lane & 7)) << 4));
        r[4 * v] = x.x; r[4 * v + 1] = x.y; r[4 * v + 2] = x.z; r[4 * v + 3] = x.w;
    }
}

// A warp's 32 features x 32 tokens (r[j] = token j of the lane's feature) of a partial tile [token][128 features] at `part` of every
// CTA of this rank in its pair, added up over the cluster's `split` pairs in the order of their pieces of K.
__device__ __forceinline__ void tmw_sum(uint32_t part, int split, uint32_t rank, int chunk, int feature, uint32_t (&r)[32])
{
    for (int s = 0; s < split; ++s) {
        const uint32_t src = ptx::map_to_cta(part, 2u * s + rank) + (uint32_t)(chunk * 32 * 512 + feature * 4);
        float x[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(x[j]) : "r"(src + 512u * j) : "memory");
#pragma unroll
        for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(s ? __uint_as_float(r[j]) + x[j] : x[j]);
    }
}

// The tile's results of 32 tokens from m0 on: bias, ReLU, residual, fp32 or MXInt store.  buf: the warp's transposing buffer (QOUT).
template <bool QOUT>
__device__ __forceinline__ void tmw_store(const TcParams &p, int m0, int n, float bias, uint8_t *buf, int lane, uint32_t (&r)[32])
{
    tmw_tail(p, m0, n, bias, r);
    if (QOUT) {
        tmw_transpose(buf, lane, r);
        store_mxint_chunk(p, m0 + lane, n - lane, r);
    } else if (n < p.N) {
        float *dst = p.y + (int64_t)m0 * p.ldy + n;
        if (m0 + 32 <= p.M) {
#pragma unroll
            for (int j = 0; j < 32; ++j) dst[(int64_t)j * p.ldy] = __uint_as_float(r[j]);
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (m0 + j < p.M) dst[(int64_t)j * p.ldy] = __uint_as_float(r[j]);
        }
    }
}

// SPLIT: K cut over the pairs of a cluster.
template <bool NIB, bool QOUT, bool SPLIT>
__global__ void __maxnreg__(80)
gemm_tmw_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_r, const TcParams p, const TmwParams wp)
{
    using Cfg = TmwCfg;
    constexpr int GROUPS = Cfg::GROUPS, RS = Cfg::RAW_STAGES, MAX_AS = Cfg::MAX_A_STAGES;
    constexpr int STEP_BYTES = NIB ? 32 : 64;                            // packed bytes of a row per K step
    constexpr int SPR = 128 / STEP_BYTES;                                // K steps per raw stage
    const bool b16 = wp.block == 16;
    const int EB = (NIB ? 16 : 8) >> (b16 ? 0 : 1);                      // exponent bytes of a row per raw stage
    const int EW = (EB >> 2) + (wp.exp_words ? 0 : 1);                   // the aligned words that hold them
    const int T = wp.tokens, stages = wp.stages, accs = Cfg::accs(T);
    const uint32_t as_shift = Cfg::a_stages(T) == 8 ? 3 : 2, as_mask = (1u << as_shift) - 1u, a_col = Cfg::a_col(T), acc_col = Cfg::acc_col(T);
    const uint32_t stage_bytes = Cfg::stage_bytes(T);
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_gen = smem_raw + (smem_base - ptx::smem_u32(smem_raw));
    const uint32_t raw_base = smem_base, exp_base = raw_base + RS * Cfg::RAW_MANT, x_base = smem_base + Cfg::RAW_BYTES, tr_base = x_base + stages * stage_bytes;
    const uint32_t bar_base = tr_base + (QOUT ? Cfg::EPI_WARPS * 4096 : 0);
    auto x_full = [&](int s) { return bar_base + 8u * s; };
    auto x_empty = [&](int s) { return bar_base + 8u * (Cfg::MAX_STAGES + s); };
    auto a_full = [&](int s) { return bar_base + 8u * (2 * Cfg::MAX_STAGES + s); };
    auto a_empty = [&](int s) { return bar_base + 8u * (2 * Cfg::MAX_STAGES + MAX_AS + s); };
    auto r_full = [&](int s) { return bar_base + 8u * (2 * Cfg::MAX_STAGES + 2 * MAX_AS + s); };
    auto r_empty = [&](int s) { return bar_base + 8u * (2 * Cfg::MAX_STAGES + 2 * MAX_AS + RS + s); };
    constexpr int ACC_BARS = 2 * Cfg::MAX_STAGES + 2 * MAX_AS + 2 * RS;
    auto t_full = [&](int a) { return bar_base + 8u * (ACC_BARS + a); };
    auto t_empty = [&](int a) { return bar_base + 8u * (ACC_BARS + 2 + a); };
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem_gen + (bar_base - smem_base) + 8 * (ACC_BARS + 4));
    volatile uint32_t *abort_flag = tmem_slot + 1;
    static_assert(8 * (ACC_BARS + 4) + 8 <= 512 && Cfg::RAW_BYTES % 1024 == 0, "barriers; the activations' tiles are aligned");

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t cta = ptx::cluster_ctarank(), rank = cta & 1u, lead = SPLIT ? cta & ~1u : 0u;      // rank 0: leader of its pair
    const bool leader = rank == 0;
    const uint16_t both = (uint16_t)(3u << lead);                        // the pair's CTAs
    const int split = SPLIT ? wp.split : 1;
    using Walk = StepWalk<SPR, GROUPS>;
    static_assert(RS > GROUPS, "what the waits for raw stages rely on (see StepWalk)");

    if (threadIdx.x == 0) {
        for (int s = 0; s < Cfg::MAX_STAGES; ++s) {
            ptx::mbar_init(x_full(s), 1);
            ptx::mbar_init(x_empty(s), 1);
        }
        for (int s = 0; s < MAX_AS; ++s) {
            ptx::mbar_init(a_full(s), 8);                                // four decoding warps of either CTA
            ptx::mbar_init(a_empty(s), 1);
        }
        for (int s = 0; s < RS; ++s) {
            ptx::mbar_init(r_full(s), 33);                               // the mantissa bytes, each producer lane's exponents
            ptx::mbar_init(r_empty(s), 4 * SPR);                         // four warps per K step
        }
        for (int a = 0; a < 2; ++a) {
            ptx::mbar_init(t_full(a), 1);
            ptx::mbar_init(t_empty(a), 2 * Cfg::EPI_WARPS);              // the epilogue warps of both CTAs
        }
        *abort_flag = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tmap_x);
        ptx::prefetch_tensormap(&tmap_r);
    }
    if (warp == 1) {
        ptx::tmem_alloc_pair(ptx::smem_u32(tmem_slot), Cfg::TMEM_COLS);
        ptx::tmem_relinquish_pair();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_sync();                                                 // the peer's barriers exist before anyone signals them
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;

    const int num_tiles = p.tiles_m * p.tiles_n;                         // tiles_m of tokens, tiles_n of 256 features
    const int pair = blockIdx.x / (2 * split), npairs = gridDim.x / (2 * split);          // (K cut: a cluster of pairs)
    // the pair's piece of K: whole raw stages; split <= their number
    const int k_all = (p.K + TC_BK - 1) / TC_BK, raws_all = (k_all + SPR - 1) / SPR, piece = SPLIT ? (int)(cta >> 1) : 0;
    const int kb0 = raws_all * piece / split * SPR, kblocks = min(k_all, raws_all * (piece + 1) / split * SPR) - kb0, raws = (kblocks + SPR - 1) / SPR;
    bool timed_out = false;
    // early: the launch in front only writes the activations' operand form, and starts this one when ITS predecessors are
    // complete: the weights may be fetched and decoded meanwhile (decoding writes tensor memory alone)
    if (!(wp.early && warp >= 2 && warp < 4 + 4 * GROUPS)) ptx::dep_wait();
    if (threadIdx.x == 0) ptx::dep_trigger();

    if (warp == 0) {
        int s = 0;
        uint32_t ph = 0;
        for (int t = pair; t < num_tiles && !timed_out; t += npairs) {
            const int m0 = (t % p.tiles_m) * T + (int)rank * (T / 2);
            for (int kb = 0; kb < kblocks; kb += 2) {
                if (!__all_sync(0xFFFFFFFFu, ptx::mbar_wait_bounded_relaxed(x_empty(s), ph ^ 1u, abort_flag, TC_WAIT_LIMIT_NS))) {
                    timed_out = true;
                    break;
                }
                if (ptx::elect_one()) {
                    const uint32_t leader_full = ptx::map_to_cta(x_full(s), lead), sx = x_base + s * stage_bytes;
                    const bool two = kb + 1 < kblocks;
                    if (leader) ptx::mbar_arrive_expect_tx(x_full(s), two ? 2 * stage_bytes : stage_bytes);
                    ptx::tma_load_2d_pair(sx, &tmap_x, (kb0 + kb) * TC_BK, m0, leader_full);
                    if (two) ptx::tma_load_2d_pair(sx + (stage_bytes >> 1), &tmap_x, (kb0 + kb + 1) * TC_BK, m0, leader_full);
                }
                if (++s == stages) { s = 0; ph ^= 1u; }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // the whole warp runs the loop, its elected lane issues (see ptx::elect_one)
        if (leader) {
            const uint32_t idesc = ptx::idesc_bf16_f32(256, T);
            const uint64_t desc0 = ptx::smem_desc_k_sw128(x_base, 0);
            const uint32_t tm = __shfl_sync(0xFFFFFFFFu, tmem_base, 0);
            int s = 0, it = 0;
            uint32_t ph = 0, step = 0;
            bool ready = false;                                          // the next steps' operands are there already
            auto wait_a = [&](uint32_t i) { return ptx::mbar_wait_bounded_relaxed(a_full(i & as_mask), (i >> as_shift) & 1u, abort_flag, TC_WAIT_LIMIT_NS); };
            auto test_a = [&](uint32_t i) { return ptx::mbar_test(a_full(i & as_mask), (i >> as_shift) & 1u); };
            for (int t = pair; t < num_tiles && !timed_out; t += npairs, ++it) {
                const int acc = accs == 2 ? it & 1 : 0;
                const uint32_t acc_ph = (uint32_t)(accs == 2 ? it >> 1 : it) & 1u;
                bool ok = ptx::mbar_wait_bounded_relaxed(t_empty(acc), acc_ph ^ 1u, abort_flag, TC_WAIT_LIMIT_NS);
                const uint32_t d_tmem = tm + (uint32_t)acc * acc_col;
                for (int kb = 0; kb < kblocks; kb += 2) {
                    const bool two = kb + 1 < kblocks;
                    if (kb == 0 || !ready) {
                        ok = ok && (ready || (wait_a(step) && (!two || wait_a(step + 1)) &&
                                              ptx::mbar_wait_bounded(x_full(s), ph, abort_flag, TC_WAIT_LIMIT_NS)));
                        if (!__all_sync(0xFFFFFFFFu, ok)) {
                            timed_out = true;
                            break;
                        }
                    }
                    ptx::tc_fence_after_sync();
                    const int cur = s;
                    const uint32_t a0 = step & as_mask, a1 = (step + 1) & as_mask;
                    if (++s == stages) { s = 0; ph ^= 1u; }
                    step += two ? 2 : 1;
                    // the answers for the next two steps arrive while the MMAs are issued
                    const bool next_two = kb + 2 < kblocks ? kb + 3 < kblocks : kblocks > 1;
                    const bool n0 = test_a(step), n1 = test_a(step + (next_two ? 1 : 0)), nx = ptx::mbar_test(x_full(s), ph);
                    if (ptx::elect_one()) {
                        const uint64_t desc = desc0 + (uint64_t)((uint32_t)cur * (stage_bytes >> 4));
#pragma unroll
                        for (int j = 0; j < TC_BK / 16; ++j)
                            ptx::mma_bf16_ts_pair(d_tmem, tm + a_col + 32u * a0 + 8u * j, desc + 2u * j, idesc, (kb | j) != 0 ? 1u : 0u);
                        ptx::mma_commit_pair(a_empty(a0), both);            // both CTAs may refill their stages
                        if (two) {
#pragma unroll
                            for (int j = 0; j < TC_BK / 16; ++j)
                                ptx::mma_bf16_ts_pair(d_tmem, tm + a_col + 32u * a1 + 8u * j, desc + (stage_bytes >> 5) + 2u * j, idesc, 1u);
                            ptx::mma_commit_pair(a_empty(a1), both);
                        }
                        ptx::mma_commit_pair(x_empty(cur), both);
                    }
                    ready = __all_sync(0xFFFFFFFFu, n0 && n1 && nx);
                }
                if (timed_out) break;
                if (ptx::elect_one()) ptx::mma_commit_pair(t_full(acc), both);
            }
        }
        __syncwarp();
    } else if (warp == 2) {
        // raw stages: 128 rows x 128 mantissa bytes in one tiled load, their exponent bytes in the background (see gemm_dec_kernel)
        ExpFeed feed(wp.w_exp, p.K / wp.block, EB, wp.exp_words);
        const bool wait_last = Walk::waits_for_last(kblocks);            // (see StepWalk)
        uint32_t ri = 0;
        for (int t = pair; t < num_tiles && !timed_out; t += npairs) {
            if (wait_last && ri && !__all_sync(0xFFFFFFFFu, ptx::mbar_wait_bounded(r_full((ri - 1) % RS), ((ri - 1) / RS) & 1u, abort_flag, TC_WAIT_LIMIT_NS))) {
                timed_out = true;
                break;
            }
            const int n0 = (t / p.tiles_m) * 256 + (int)rank * Cfg::BN;
            feed.rows(wp.w_exp, n0, p.N, wp.w_rows2, lane);
            for (int i = 0; i < raws; ++i, ++ri) {
                const int s = ri % RS;
                const bool ok = ptx::mbar_wait_bounded(r_empty(s), ((ri / RS) & 1u) ^ 1u, abort_flag, TC_WAIT_LIMIT_NS);
                if (!__all_sync(0xFFFFFFFFu, ok)) {
                    timed_out = true;
                    break;
                }
                const int kb = kb0 + i * SPR, b0 = kb * (b16 ? 4 : 2);
                if (lane == 0) {
                    ptx::fence_proxy_async_smem();
                    ptx::mbar_arrive_expect_tx(r_full(s), Cfg::RAW_MANT);
                    ptx::tma_load_2d(raw_base + s * Cfg::RAW_MANT, &tmap_r, kb * STEP_BYTES, n0, r_full(s));      // outside the matrix: zeros
                }
                feed.copy(exp_base + s * Cfg::RAW_EXP, b0, lane);
                cp_async_arrive(r_full(s));
            }
        }
    } else if (warp >= 4 && warp < 4 + 4 * GROUPS) {
        // a lane a row, both halves of the step, straight into the row's 32 columns of the stage
        const int g = (warp - 4) >> 2, quad = warp & 3, r = 32 * quad + lane;
        // Shared addresses are 32-bit offsets whose parts are worked out once: of the 260 instructions that a step cost a warp, 110
        // decode (240 now; 512 x 4096 x 11008 with an MXInt8 result, tiles of 192 tokens, 55.3 -> 53.3 us; at 224 tokens the MMAs bind).
        const uint32_t mrow = raw_base - smem_base + r * 128, swz = (uint32_t)(r & 7) << 4, ebase = exp_base - smem_base + r * (4 * EW);
        const uint32_t dst = tmem_base + ((uint32_t)(quad * 32) << 16) + a_col, a_full_lead = ptx::map_to_cta(a_full(0), lead);
        const bool e_word = b16 && wp.exp_words;
        uint32_t erow = ebase;
        Walk at{g, pair, 0, (uint32_t)g};
        auto row_exps = [&]() {                                          // where the tile's exponent bytes of this row start
            const int n = min((at.tile / p.tiles_m) * 256 + (int)rank * Cfg::BN + r, p.N - 1);
            erow = ebase + ((uint32_t)reinterpret_cast<uintptr_t>(wp.w_exp + (int64_t)(n >> wp.w_rows2) * (p.K / wp.block)) & 3u);
        };
        auto settle = [&]() {
            if (at.kb < kblocks) return;
            at.settle(kblocks, raws, npairs);
            if (at.tile < num_tiles) row_exps();
        };
        row_exps();
        settle();
        // Each barrier is looked at well before its answer is needed: waiting for one that is long complete takes 130 clocks, of
        // which a step of this loop had three in about 1500.
        bool there = false;                                              // the raw stage is known to be full
        uint32_t ri = at.raw();                                          // raw stages before this step's
        while (at.tile < num_tiles) {
            const uint32_t j = (uint32_t)at.kb % SPR, a = at.step & as_mask, a_ph = ((at.step >> as_shift) & 1u) ^ 1u, rs = ri % RS;
            const bool last = at.kb == kblocks - 1;
            if (!there && !__all_sync(0xFFFFFFFFu, (!Walk::ASKS_EMPTY || ptx::mbar_wait_bounded(r_empty(rs), ((ri / RS) & 1u) ^ 1u, abort_flag, TC_WAIT_LIMIT_NS)) &&
                                                   ptx::mbar_wait_bounded(r_full(rs), (ri / RS) & 1u, abort_flag, TC_WAIT_LIMIT_NS))) {
                timed_out = true;
                break;
            }
            bool free = ptx::mbar_test(a_empty(a), a_ph);
            // (the exponents of all 32 rows: one path per warp)
            const uint8_t *ex = smem_gen + (erow + rs * Cfg::RAW_EXP);
            const uint32_t e4 = e_word ? *reinterpret_cast<const uint32_t *>(ex + 4 * j) : step_exps(ex, (int)j, b16, wp.exp_words);
            const uint32_t chunks = mrow + rs * Cfg::RAW_MANT + ((j * (uint32_t)STEP_BYTES) ^ swz);      // 16-byte chunk c of the row: chunks ^ 16 c
            auto load = [&](int h, uint4 (&m)[NIB ? 1 : 2]) {
#pragma unroll
                for (int q = 0; q < (NIB ? 1 : 2); ++q) m[q] = *reinterpret_cast<const uint4 *>(smem_gen + (chunks ^ (uint32_t)((NIB ? h : 2 * h + q) << 4)));
            };
            auto store = [&](int h, const uint32_t (&o)[4][4]) {
                if (h == 0) {                                            // the stage is needed only now
                    free = __all_sync(0xFFFFFFFFu, free) ||
                           __all_sync(0xFFFFFFFFu, ptx::mbar_wait_bounded_relaxed(a_empty(a), a_ph, abort_flag, TC_WAIT_LIMIT_NS));
                    ptx::tc_fence_after_sync();
                }
                ptx::tmem_st_32x16(dst + 32u * a + 16u * h, o);
            };
            uint4 m[2][NIB ? 1 : 2];
            load(0, m[0]);
            load(1, m[1]);
            if (__all_sync(0xFFFFFFFFu, exps_plain(e4, wp.w_bits))) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t o[4][4];
                    decode32_plain<NIB>(m[h], (e4 >> (16 * h)) & 0xFFu, (e4 >> (16 * h + 8)) & 0xFFu, wp.w_bits, o);
                    store(h, o);
                }
            } else {
#pragma unroll 1
                for (int h = 0; h < 2; ++h) {                            // (read again: an array indexed by a loop would live in memory)
                    uint4 again[NIB ? 1 : 2];
                    uint32_t o[4][4];
                    load(h, again);
                    decode32_perm<NIB>(again, (e4 >> (16 * h)) & 0xFFu, (e4 >> (16 * h + 8)) & 0xFFu, wp.w_bits, o);
                    store(h, o);
                }
            }
            if (!free) {
                timed_out = true;
                break;
            }
            at.step += GROUPS;
            at.kb += GROUPS;
            settle();
            ri = at.raw();
            bool next = true;                                            // (not used behind the last tile)
            if (Walk::ASKS_EMPTY) next = ptx::mbar_test(r_empty(ri % RS), ((ri / RS) & 1u) ^ 1u);
            next = ptx::mbar_test(r_full(ri % RS), (ri / RS) & 1u) && next;
            ptx::tmem_st_wait();
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) {
                ptx::mbar_arrive_cluster_relaxed(a_full_lead + 8u * a);
                ptx::mbar_arrive(r_empty(rs));
                if (last)                                                // the steps that the tile's last raw stage does not have
                    for (int x = kblocks; x < raws * SPR; ++x) ptx::mbar_arrive(r_empty(rs));
            }
            there = __all_sync(0xFFFFFFFFu, next);
        }
    } else if (warp >= 4 + 4 * GROUPS) {
        const int quad = warp & 3, half = (warp - 4 - 4 * GROUPS) >> 2;
        int it = 0;
        for (int t = pair; t < num_tiles && !timed_out; t += npairs, ++it) {
            const int acc = accs == 2 ? it & 1 : 0;
            const uint32_t acc_ph = (uint32_t)(accs == 2 ? it >> 1 : it) & 1u;
            const int n = (t / p.tiles_m) * 256 + (int)rank * Cfg::BN + quad * 32 + lane, m0 = (t % p.tiles_m) * T;
            const float bias = p.ex_bias && n < p.N ? __ldg(p.ex_bias + n) : 0.f;
            const bool ok = ptx::mbar_wait_bounded_relaxed(t_full(acc), acc_ph, abort_flag, TC_WAIT_LIMIT_NS);
            if (!__all_sync(0xFFFFFFFFu, ok)) {
                timed_out = true;
                break;
            }
            ptx::tc_fence_after_sync();
            const uint32_t src = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)acc * acc_col;
#pragma unroll 1
            for (int c = 32 * half; c < T; c += 64) {
                if (m0 + c >= p.M || n - lane >= p.N) continue;          // warp-uniform
                uint32_t r[32];
                ptx::tmem_ld_32x32(src + (uint32_t)c, r);
                ptx::tmem_ld_wait();
                if (SPLIT) {
                    // the partial tile, [token][feature], over the stages: all loads have landed and been used when t_full completes
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        *reinterpret_cast<uint32_t *>(smem_gen + (c + j) * 512 + (quad * 32 + lane) * 4) = r[j];
                } else {
                    tmw_store<QOUT>(p, m0 + c, n, bias, smem_gen + (tr_base - smem_base) + 4096 * (warp - 4 - 4 * GROUPS), lane, r);
                }
            }
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive_cluster_relaxed(ptx::map_to_cta(t_empty(acc), lead));
        }
    }

    if (timed_out) {
        *abort_flag = 1;
        atomicOr(p.status, STATUS_TIMEOUT_BIT);
        const uint64_t t0 = ptx::globaltimer_ns();
        while (ptx::globaltimer_ns() - t0 < 100000ull) __nanosleep(1000);
    }
    if (SPLIT) {
        __syncwarp();
        ptx::cluster_sync();                                             // every partial tile is in place
        if (warp >= 4 + 4 * GROUPS) {
            const int n0 = (pair / p.tiles_m) * 256 + (int)rank * Cfg::BN, m0 = (pair % p.tiles_m) * T;
            // quarter u & 3 of the features of tokens 32 (u >> 2) ..: dealt to the epilogue warps of all pairs
            for (int u = piece + split * (warp - 4 - 4 * GROUPS); u < T / 8; u += split * Cfg::EPI_WARPS) {
                const int c = u >> 2, f = (u & 3) * 32 + lane, n = n0 + f;
                if (m0 + 32 * c >= p.M || n - lane >= p.N) continue;     // warp-uniform
                uint32_t r[32];
                tmw_sum(smem_base, split, rank, c, f, r);
                tmw_store<QOUT>(p, m0 + 32 * c, n, p.ex_bias && n < p.N ? __ldg(p.ex_bias + n) : 0.f,
                                smem_gen + (tr_base - smem_base) + 4096 * (warp - 4 - 4 * GROUPS), lane, r);
            }
        }
        __syncwarp();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_sync();          // the peer no longer signals this CTA's barriers, no MMA reads its memory
    if (warp == 1) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc_pair(tmem_base, Cfg::TMEM_COLS);
    }
}

}  // namespace mx
