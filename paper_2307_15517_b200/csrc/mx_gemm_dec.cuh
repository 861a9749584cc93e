// Tensor-core MXInt product for up to 384 rows (a short prompt, a batch of decoding sequences): the packed weights are decoded
// inside the kernel, once.  Sec. 3.2 operator on exactly decoded operands, as mx_gemm_tc.cuh.
//
// At these sizes a layer's time is what its weights cost: a pass in front writes them out at two bytes per element and the
// product's CTAs fetch those once per 128 rows, an SM taking in 58 bytes per clock.  Here a CTA owns 128 columns and ALL rows
// -- P panels of 128, an accumulator in tensor memory each -- and a piece of K (a cluster shares the tile, the partial tiles are
// added through distributed shared memory as in mx_gemm_splitk.cuh); per K step of 64 it fetches P * 16 KB of A and 4 (8) KB of
// packed weights, whose decoded tile serves all P panels.
//   warp 0      : A tiles by TMA
//   warp 1      : tensor-memory allocation, MMA issue
//   warp 2      : packed weights: 128 rows x 128 bytes by TMA, exponent bytes by background copies (plain loads in flight would be
//                 waited for at every proxy fence that publishes a decoded step)
//   warps 4..15 : three groups that decode every third K step each -- a step is a chain of a wait, a shared-memory read, the
//                 conversion, the stores, a proxy fence and an arrival, about 0.6 us whatever its size -- then the partial tiles,
//                 reduction and epilogue
// Bound by shared memory with three panels (per step 48 + 20 KB written, 96 + 4 KB read at 128 bytes per clock), by the decoding
// warps and an SM's intake with one, and up to about eight steps per CTA by the chain from the first fetch to the last reduced
// value.  Whole calls, M x K x N, 8/4 bits, behind a pass over the weights / here (us): 128 x 4096 x 4096 19.5 / 14.7,
// 128 x 11008 x 4096 40.1 / 24.4, 256 x 8192 x 8192 72 / 44, 384 x 8192 x 8192 91 / 59.  Tried and slower: two K steps per proxy fence
// and group with four stages of A in place of seven (0.1 to 0.5 us), a ring of A in panels instead of K steps.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "mx_gemm_splitk.cuh"
#include "mx_gemm_tc.cuh"
#include "mx_gemv_mma.cuh"
#include "mx_ptx.cuh"

namespace mx {

struct DecCfg {
    static constexpr int BN = 128, MAX_P = 3, MAX_SPLIT = 8, MAX_STAGES = 7;
    static constexpr int GROUPS = 3, RAW_STAGES = 3;                    // decode groups, each with a W stage; raw stages
    static constexpr int THREADS = 32 * (4 + 4 * GROUPS);
    static constexpr uint32_t PANEL_BYTES = TC_BM * TC_BK * 2, W_BYTES = BN * TC_BK * 2;
    static constexpr uint32_t RAW_MANT = BN * 128, RAW_EXP = BN * 20;   // 128 mantissa bytes and the words of at most 16 exponent bytes per row
    static constexpr int stages(int P) { return P == 1 ? 7 : P == 2 ? 3 : 2; }                   // of A: what fits
    static constexpr uint32_t smem_bytes(int P)
    {
        return stages(P) * P * PANEL_BYTES + GROUPS * W_BYTES + RAW_STAGES * (RAW_MANT + RAW_EXP) + 512 + 1024;
    }
};
static_assert(DecCfg::smem_bytes(1) <= 227 * 1024 && DecCfg::smem_bytes(2) <= 227 * 1024 && DecCfg::smem_bytes(3) <= 227 * 1024, "shared memory");
static_assert(DecCfg::smem_bytes(1) >= 1 * 65536 + 1536 && DecCfg::smem_bytes(2) >= 2 * 65536 + 1536 && DecCfg::smem_bytes(3) >= 3 * 65536 + 1536,
              "the partial tiles reuse the stages");

struct DecParams {
    const uint8_t *w_exp;
    int w_bits, w_rows2, block;
    int split;
    int early;                // 1: the launch in front is this call's activation pass
    int exp_words;            // 1: every row's exponent bytes start at a whole word
};

template <int P, bool NIB, bool QOUT>
__global__ void __maxnreg__(128)
gemm_dec_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_r, const TcParams p, const DecParams dp)
{
    using Cfg = DecCfg;
    constexpr int STAGES = Cfg::stages(P), GROUPS = Cfg::GROUPS, RS = Cfg::RAW_STAGES;
    constexpr uint32_t A_BYTES = P * Cfg::PANEL_BYTES;
    constexpr int STEP_BYTES = NIB ? 32 : 64;                            // packed bytes of a row per K step
    constexpr int SPR = 128 / STEP_BYTES;                                // K steps per raw stage
    const bool b16 = dp.block == 16;
    const int EB = (NIB ? 16 : 8) >> (b16 ? 0 : 1);                      // exponent bytes of a row per raw stage
    const int EW = (EB >> 2) + (dp.exp_words ? 0 : 1);                   // the aligned words that hold them
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_gen = smem_raw + (smem_base - ptx::smem_u32(smem_raw));
    const uint32_t w_base = smem_base + STAGES * A_BYTES, raw_base = w_base + GROUPS * Cfg::W_BYTES, exp_base = raw_base + RS * Cfg::RAW_MANT;
    const uint32_t bar_base = exp_base + RS * Cfg::RAW_EXP;
    auto a_full = [&](int s) { return bar_base + 8u * s; };
    auto a_empty = [&](int s) { return bar_base + 8u * (Cfg::MAX_STAGES + s); };
    auto w_full = [&](int g) { return bar_base + 8u * (2 * Cfg::MAX_STAGES + g); };
    auto w_empty = [&](int g) { return bar_base + 8u * (2 * Cfg::MAX_STAGES + GROUPS + g); };
    auto r_full = [&](int s) { return bar_base + 8u * (2 * Cfg::MAX_STAGES + 2 * GROUPS + s); };
    auto r_empty = [&](int s) { return bar_base + 8u * (2 * Cfg::MAX_STAGES + 2 * GROUPS + RS + s); };
    const uint32_t done_bar = bar_base + 8u * (2 * Cfg::MAX_STAGES + 2 * GROUPS + 2 * RS);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem_gen + (done_bar + 8u - smem_base));
    volatile uint32_t *abort_flag = tmem_slot + 1;
    constexpr uint32_t TMEM_COLS = P == 1 ? 128 : P == 2 ? 256 : 512;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int split = dp.split, rank = (int)ptx::cluster_ctarank(), tile = (int)blockIdx.x / split;

    if (threadIdx.x == 0) {
        for (int s = 0; s < Cfg::MAX_STAGES; ++s) {
            ptx::mbar_init(a_full(s), 1);
            ptx::mbar_init(a_empty(s), 1);
        }
        for (int g = 0; g < GROUPS; ++g) {
            ptx::mbar_init(w_full(g), 4);                                // the group's warps
            ptx::mbar_init(w_empty(g), 1);
        }
        for (int s = 0; s < RS; ++s) {
            ptx::mbar_init(r_full(s), 33);                               // the mantissa bytes, each producer lane's exponents
            ptx::mbar_init(r_empty(s), 4 * SPR);                         // four warps per K step
        }
        ptx::mbar_init(done_bar, 1);
        *abort_flag = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tmap_a);
        ptx::prefetch_tensormap(&tmap_r);
    }
    if (warp == 1) {
        ptx::tmem_alloc(ptx::smem_u32(tmem_slot), TMEM_COLS);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;

    // pieces of whole pairs of K steps (their exponent bytes start at whole words); split <= pairs: every CTA has a step
    const int kblocks = (p.K + TC_BK - 1) / TC_BK, pairs = (kblocks + 1) >> 1;
    const int kb0 = 2 * (pairs * rank / split), kb1 = min(kblocks, 2 * (pairs * (rank + 1) / split)), steps = kb1 - kb0;
    const int n0 = tile * Cfg::BN;
    bool timed_out = false;
    // early: the launch in front only writes the activations' operand form, and starts this one when ITS predecessors are
    // complete: the weights may be fetched and decoded meanwhile
    if (!(dp.early && (warp == 2 || warp >= 4))) ptx::dep_wait();
    if (threadIdx.x == 0) ptx::dep_trigger();

    if (warp == 0) {
        int s = 0;
        uint32_t ph = 0;
        for (int i = 0; i < steps; ++i) {
            if (!__all_sync(0xFFFFFFFFu, ptx::mbar_wait_bounded(a_empty(s), ph ^ 1u, abort_flag, TC_WAIT_LIMIT_NS))) {
                timed_out = true;
                break;
            }
            if (ptx::elect_one()) {
                ptx::mbar_arrive_expect_tx(a_full(s), A_BYTES);
#pragma unroll
                for (int q = 0; q < P; ++q)
                    ptx::tma_load_2d(smem_base + s * A_BYTES + q * Cfg::PANEL_BYTES, &tmap_a, (kb0 + i) * TC_BK, q * TC_BM, a_full(s));
            }
            if (++s == STAGES) { s = 0; ph ^= 1u; }
        }
        __syncwarp();
    } else if (warp == 1) {
        constexpr uint32_t idesc = ptx::idesc_bf16_f32(TC_BM, Cfg::BN);
        const uint32_t tm = __shfl_sync(0xFFFFFFFFu, tmem_base, 0);
        const uint64_t desc_a = ptx::smem_desc_k_sw128(smem_base, 0), desc_w = ptx::smem_desc_k_sw128(w_base, 0);
        int s = 0, g = 0;
        uint32_t ph = 0, gph = 0;
        bool ready = false;                                              // the next step's operands are there already
        for (int i = 0; i < steps; ++i) {
            if (!ready && !__all_sync(0xFFFFFFFFu, ptx::mbar_wait_bounded(a_full(s), ph, abort_flag, TC_WAIT_LIMIT_NS) &&
                                                   ptx::mbar_wait_bounded(w_full(g), gph, abort_flag, TC_WAIT_LIMIT_NS))) {
                timed_out = true;
                break;
            }
            ptx::tc_fence_after_sync();
            const int cur = s, curg = g;
            if (++s == STAGES) { s = 0; ph ^= 1u; }
            if (++g == GROUPS) { g = 0; gph ^= 1u; }
            const bool ahead_a = ptx::mbar_test(a_full(s), ph), ahead_w = ptx::mbar_test(w_full(g), gph);      // answers arrive meanwhile
            if (ptx::elect_one()) {
                const uint64_t da = desc_a + (uint64_t)((uint32_t)cur * (A_BYTES >> 4)), dw = desc_w + (uint64_t)((uint32_t)curg * (Cfg::W_BYTES >> 4));
#pragma unroll
                for (int q = 0; q < P; ++q)
#pragma unroll
                    for (int j = 0; j < TC_BK / 16; ++j)
                        ptx::mma_bf16_ss(tm + 128u * q, da + (uint32_t)(q * (Cfg::PANEL_BYTES >> 4) + 2 * j), dw + 2u * j, idesc, (i | j) != 0 ? 1u : 0u);
                ptx::mma_commit(a_empty(cur));
                ptx::mma_commit(w_empty(curg));
            }
            ready = __all_sync(0xFFFFFFFFu, ahead_a && ahead_w);
        }
        if (!timed_out && ptx::elect_one()) ptx::mma_commit(done_bar);
        __syncwarp();
    } else if (warp == 2) {
        // raw stages: 128 rows x 128 mantissa bytes in one tiled load, their exponent bytes in the background
        const int nb = p.K / dp.block, raws = (steps + SPR - 1) / SPR;
        for (int i = 0; i < raws; ++i) {
            const int s = i % RS;
            const bool ok = ptx::mbar_wait_bounded(r_empty(s), ((uint32_t)(i / RS) & 1u) ^ 1u, abort_flag, TC_WAIT_LIMIT_NS);
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
            uint8_t *dx = smem_gen + (exp_base - smem_base) + s * Cfg::RAW_EXP;
            // whole words from the one that holds the row's first byte on, the row's end cut off (zeros): rows at odd addresses byte
            // by byte, in plain loads, made this warp the kernel's slowest (128 x 2080 x 11008, M x K x N, 8/4 in blocks of 16: 45.9 us
            // against 24.7; 33 x 11040 x 11008, 8/8, 393 against 95)
            for (int wi = lane; wi < Cfg::BN * EW; wi += 32) {
                const int r = wi / EW;
                const uint8_t *row = dp.w_exp + (int64_t)(min(n0 + r, p.N - 1) >> dp.w_rows2) * nb;
                const uint32_t skip = (uint32_t)reinterpret_cast<uintptr_t>(row) & 3u;         // (b0 is a multiple of 4)
                const int at = b0 + (wi - r * EW) * 4 - (int)skip, valid = min(nb - at, 4);
                cp_async4(ptx::smem_u32(dx) + wi * 4, row + (valid > 0 ? at : -(int)skip), max(valid, 0));
            }
            cp_async_arrive(r_full(s));
        }
    } else if (warp >= 4) {
        // group g fills W stage g with the K steps g, g + 3, ...: a lane a row, both halves of the step.  Eight rows per phase of
        // a 16-byte access, chunks swizzled by the row: no bank conflicts
        const int g = (warp - 4) >> 2, r = 32 * (warp & 3) + lane;
        const uint8_t *mrow = smem_gen + (raw_base - smem_base) + r * 128, *erow = smem_gen + (exp_base - smem_base) + r * (4 * EW) +
                             ((uint32_t)reinterpret_cast<uintptr_t>(dp.w_exp + (int64_t)(min(n0 + r, p.N - 1) >> dp.w_rows2) * (p.K / dp.block)) & 3u);
        uint8_t *dst = smem_gen + (w_base - smem_base) + g * Cfg::W_BYTES + (r >> 3) * 1024 + (r & 7) * 128;
        // each barrier is looked at well before its answer is needed: waiting for one that is long complete takes 130 clocks
        bool there = false;                                              // the raw stage is known to be full
        for (int i = g; i < steps; i += GROUPS) {
            const int j = i % SPR, rs = i / SPR % RS;
            const uint32_t w_ph = ((uint32_t)(i / GROUPS) & 1u) ^ 1u;
            if (!there && !__all_sync(0xFFFFFFFFu, ptx::mbar_wait_bounded(r_full(rs), (uint32_t)(i / SPR / RS) & 1u, abort_flag, TC_WAIT_LIMIT_NS))) {
                timed_out = true;
                break;
            }
            bool free = ptx::mbar_test(w_empty(g), w_ph);
            // (the exponents of all 32 rows: one path per warp)
            const uint32_t e4 = step_exps(erow + rs * Cfg::RAW_EXP, j, b16, dp.exp_words);
            auto load = [&](int h, uint4 (&m)[NIB ? 1 : 2]) {
#pragma unroll
                for (int q = 0; q < (NIB ? 1 : 2); ++q) {
                    const int c = NIB ? 2 * j + h : 4 * j + 2 * h + q;                        // 16-byte chunk of the row's 128 bytes
                    m[q] = *reinterpret_cast<const uint4 *>(mrow + rs * Cfg::RAW_MANT + ((c ^ (r & 7)) << 4));
                }
            };
            auto store = [&](int h, const uint32_t (&o)[4][4]) {
                if (h == 0)                                              // the stage is needed only now
                    free = __all_sync(0xFFFFFFFFu, free) ||
                           __all_sync(0xFFFFFFFFu, ptx::mbar_wait_bounded(w_empty(g), w_ph, abort_flag, TC_WAIT_LIMIT_NS));
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    *reinterpret_cast<uint4 *>(dst + (((h * 4 + q) ^ (r & 7)) << 4)) = make_uint4(o[q][0], o[q][1], o[q][2], o[q][3]);
            };
            uint4 m[2][NIB ? 1 : 2];
            load(0, m[0]);
            load(1, m[1]);
            if (__all_sync(0xFFFFFFFFu, exps_plain(e4, dp.w_bits))) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t o[4][4];
                    decode32_plain<NIB>(m[h], (e4 >> (16 * h)) & 0xFFu, (e4 >> (16 * h + 8)) & 0xFFu, dp.w_bits, o);
                    store(h, o);
                }
            } else {
#pragma unroll 1
                for (int h = 0; h < 2; ++h) {                            // (read again: an array indexed by a loop would live in memory)
                    uint4 again[NIB ? 1 : 2];
                    uint32_t o[4][4];
                    load(h, again);
                    decode32_perm<NIB>(again, (e4 >> (16 * h)) & 0xFFu, (e4 >> (16 * h + 8)) & 0xFFu, dp.w_bits, o);
                    store(h, o);
                }
            }
            if (!free) {
                timed_out = true;
                break;
            }
            const int in = i + GROUPS;
            const bool next = in < steps && ptx::mbar_test(r_full(in / SPR % RS), (uint32_t)(in / SPR / RS) & 1u);
            ptx::fence_proxy_async_smem();                               // the decoded rows -> visible to the MMA
            __syncwarp();
            if (lane == 0) {
                ptx::mbar_arrive(w_full(g));
                ptx::mbar_arrive(r_empty(rs));
            }
            there = __all_sync(0xFFFFFFFFu, next);
        }
        if (dp.early) ptx::dep_wait();                                   // before the results are written
        // the partial tiles: tensor memory -> this CTA's shared memory.  All its loads have landed, the raw stages are consumed
        // and all its MMAs have read their operands when done_bar completes.
        const bool ok = !timed_out && ptx::mbar_wait_bounded(done_bar, 0, abort_flag, TC_WAIT_LIMIT_NS);
        if (__all_sync(0xFFFFFFFFu, ok)) {
            ptx::tc_fence_after_sync();
            const int quad = warp & 3, row = quad * 32 + lane;
#pragma unroll 1
            for (int c = g; c < 4 * P; c += GROUPS) {                    // chunk c & 3 of panel c >> 2
                uint32_t x[32];
                ptx::tmem_ld_32x32(tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(32 * c), x);
                ptx::tmem_ld_wait();
#pragma unroll
                for (int v = 0; v < 8; ++v)
                    *reinterpret_cast<uint4 *>(smem_gen + splitk_offset(c, row, v)) = make_uint4(x[4 * v], x[4 * v + 1], x[4 * v + 2], x[4 * v + 3]);
            }
            ptx::tc_fence_before_sync();
        } else {
            timed_out = true;
        }
    }
    if (timed_out) {
        *abort_flag = 1;
        atomicOr(p.status, STATUS_TIMEOUT_BIT);
        const uint64_t t0 = ptx::globaltimer_ns();
        while (ptx::globaltimer_ns() - t0 < 100000ull) __nanosleep(1000);
    }
    __syncwarp();
    ptx::cluster_sync();                                                 // every partial tile is in place
    if (warp >= 4) splitk_reduce<true, QOUT>(p, smem_gen, smem_base, split, rank, 4 * P, 4, 0, n0, warp - 4, 4 * GROUPS, lane);
    __syncwarp();
    ptx::tc_fence_before_sync();
    ptx::cluster_sync();                                                 // nobody reads this CTA's partial tiles any more
    if (warp == 1) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(tmem_base, TMEM_COLS);
    }
}

}  // namespace mx
