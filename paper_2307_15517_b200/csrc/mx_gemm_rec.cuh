// MXInt product on the tensor pipe's block-scaled 8-bit path, CTA pairs (Sec. 3.2: the MXInt dot-product operator
// applies the shared exponent once per block; tcgen05.mma.kind::mxf8f6f4.block_scale is that operator in silicon).
// Operands are records (mx_records.cuh): mantissas of up to 5 bits on both sides, blocks of 16 and of 32.  Products are
// exact, the 32 products of an MMA step are summed with the scale 2^(Ea+Ew) and accumulate in fp32 in tensor memory, as
// in the bf16 kernels; the 8-bit pipe runs at twice their rate on half their operand bytes.  (Wider mantissas split into
// two E4M3 planes take two MMAs: measured, and no faster than bf16: 2048 x 12288 x 4096 188 against 192 us, 2048^3 28
// against 24.)
//
// Two CTAs on neighbouring SMs (a cluster of two) share one 256 x 256 output tile, K step 128: each holds one record
// of A and one of W per step, plus the scales of its own A rows and of all 256 rows of W (the pair's MMA reads the W
// scales from both CTAs' tensor memory).  The warp roles and barriers are those of mx_gemm_tc2.cuh:
//   warp 0      : TMA producer (in both CTAs; bytes are counted on the leader's barrier)
//   warp 1      : tensor-memory allocation (both CTAs), scale copies and MMA issue (leader only)
//   warps 2..9  : epilogue of the CTA's own 128 rows, two warps per TMEM lane quarter
// What bounds it: the tensor pipe, 0.28 us per 256 x 256 x 128 step and pair against the pipe's own 0.26 (0.36 while one lane issued,
// which was the bound then), with 64 KB of operands per step (17 TB/s over the chip); on few tiles per pair ramp and drain.
//
// Tensor memory: 512 columns cannot hold two accumulators of 256 and the scales.  The accumulators overlap by 32
// columns ([0, 256) and [224, 480)), the last 32 columns hold two sets of scales.  The epilogue drains the shared
// columns first and then lets the next tile's MMAs start, so what is exposed between two tiles is one 32-column read.
//
// Wide steps (the flag bytes of one of the step's four records are not all zero: some row's blocks were too far apart for
// one scale per record): every 32 k take two MMAs, one per half.  The operands' second k-chunk of 16 is then a panel of
// zeros in shared memory -- without swizzle the distance between the two chunks of an MMA is a free field of the
// descriptor -- and each half has its own scales: exact for any exponents, at the cost of twice the MMAs in these steps.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "mx_gemm_tc.cuh"
#include "mx_gemm_tc8.cuh"
#include "mx_ptx.cuh"
#include "mx_records.cuh"

namespace mx {

struct RecCfg {
    static constexpr int BN = 256;                        // pair tile: 256 x 256
    static constexpr int STAGES = 6;
    static constexpr uint32_t W_OFF = REC_BYTES;                            // A record, W record, then the scales:
    static constexpr uint32_t SFA_OFF = W_OFF + REC_BYTES;                  // own rows of A; both panels of W
    static constexpr uint32_t SFW_OFF = SFA_OFF + REC_SFW_BYTES;
    static constexpr uint32_t STAGE_BYTES = SFW_OFF + 2 * REC_SFW_BYTES;    // 35 KB
    static constexpr int EPI_WARPS = 8;
    static constexpr int THREADS = 64 + 32 * EPI_WARPS;
    static constexpr uint32_t ZERO_BYTES = REC_ROWS * 16;                   // one k-chunk of zeros
    static constexpr uint32_t BAR_BYTES = 256;
    static constexpr uint32_t SMEM_BYTES = STAGES * STAGE_BYTES + ZERO_BYTES + BAR_BYTES + 1024;
    static constexpr uint32_t TMEM_COLS = 512;
    static constexpr uint32_t ACC_STEP = 224;             // first column of the second accumulator
    static constexpr uint32_t SF_COL = 480;               // scale columns: two sets of 4 (A) + 8 (W)
    static constexpr uint32_t SF_SET = 12;
};
static_assert(RecCfg::SMEM_BYTES <= 227 * 1024, "shared memory of the record kernel");

// K-major operand without swizzle: 8 rows x 16 bytes are 128 contiguous bytes, groups of 8 rows follow each other,
// `lbo` is the distance of the MMA's second k-chunk from its first.
__device__ __forceinline__ uint64_t smem_desc_rec(uint32_t addr, uint32_t lbo)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)(128u >> 4) << 32;
    d |= (uint64_t)1 << 46;                   // descriptor version for tcgen05
    return d;
}
__device__ __forceinline__ void tmem_cp_32x128b_warpx4_pair(uint32_t taddr, uint64_t sdesc)
{
    asm volatile("tcgen05.cp.cta_group::2.32x128b.warpx4 [%0], %1;" ::"r"(taddr), "l"(sdesc) : "memory");
}
__device__ __forceinline__ void mma_mxf8_ss_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                                 uint32_t sfa_tmem, uint32_t sfb_tmem, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale [%0], %1, %2, %3, [%5], [%6], p;\n\t}"
        :
        : "r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(sfa_tmem), "r"(sfb_tmem)
        : "memory");
}

// Tensor maps over the operands' arrays: records as rows of 1 KB (box: one record), scales as rows of 512 B, half-block
// scales as rows of 1 KB (box: one panel of A, two of W).
struct RecMaps { CUtensorMap a, w, sa, sw, sa_wide, sw_wide; };

struct RecParams {
    const uint8_t *flags_a, *flags_w;        // [panels][kblocks][16]
    int panels_a, panels_w;
    int panels_sa, panels_sw;                // panels in the scale arrays
};

// The residual values of a warp's 32 x 32 chunk in the fragment shape, fetched one chunk ahead of their use.
struct FragTail { float2 v[2][2][4]; };

__device__ __forceinline__ void frag_tail_fetch(const TcParams &p, int rows0, int n, int lane, FragTail &t)
{
    if (!p.residual) return;
    const bool vec = (p.ldr & 1) == 0 && (reinterpret_cast<uintptr_t>(p.residual) & 7) == 0;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int row = rows0 + 16 * h + 8 * u + (lane >> 2);
            const float *src = p.residual + (int64_t)row * p.ldr;
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const int c = n + 8 * g + 2 * (lane & 3);
                float2 r = make_float2(0.f, 0.f);
                if (row < p.M && c + 1 < p.N && vec) {
                    r = __ldg(reinterpret_cast<const float2 *>(src + c));
                } else if (row < p.M) {
                    if (c < p.N) r.x = __ldg(src + c);
                    if (c + 1 < p.N) r.y = __ldg(src + c + 1);
                }
                t.v[h][u][g] = r;
            }
        }
}

// fp32 result of a warp's 32 x 32 chunk from the fragment shape: (+ bias) and, with TAIL, the activation and the residual,
// in the order of tail_apply.  Four neighbouring lanes write one 32-byte sector where rows of y are 8-byte aligned.
template <bool TAIL>
__device__ __forceinline__ void frag_store(const TcParams &p, const uint32_t (&r)[2][16], const FragTail &t, int rows0, int n, int lane)
{
    if (n >= p.N || rows0 >= p.M) return;                  // warp-uniform
    const float *bias = TAIL ? p.ex_bias : p.bias;
    // the sectors of a row go out one after the other (rows innermost instead: 2048^3 20.5 against 18.8 us)
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const int c = n + 8 * g + 2 * (lane & 3);
            float2 b = make_float2(0.f, 0.f);
            if (bias) {
                if (c + 1 < p.N) b = __ldg(reinterpret_cast<const float2 *>(bias + c));
                else if (c < p.N) b.x = __ldg(bias + c);
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int row = rows0 + 16 * h + 8 * u + (lane >> 2);
                if (row >= p.M || c >= p.N) continue;
                float2 v = make_float2(__uint_as_float(r[h][4 * g + 2 * u]), __uint_as_float(r[h][4 * g + 2 * u + 1]));
                if (bias) { v.x += b.x; v.y += b.y; }
                if (TAIL) {
                    if (p.relu) {                                        // NaN stays NaN
                        v.x = v.x < 0.f ? 0.f : v.x;
                        v.y = v.y < 0.f ? 0.f : v.y;
                    }
                    if (p.residual) { v.x += t.v[h][u][g].x; v.y += t.v[h][u][g].y; }
                }
                float *dst = p.y + (int64_t)row * p.ldy + c;
                if (c + 1 < p.N && p.frag_store) {
                    *reinterpret_cast<float2 *>(dst) = v;
                } else {
                    dst[0] = v.x;
                    if (c + 1 < p.N) dst[1] = v.y;
                }
            }
        }
}

// Which of 32 K steps (from 32 * kg on) of a tile are wide: every lane looks one step up, in the flag bytes of the tile's
// four records.  The loads are issued by `fetch` and first touched by `mask`, 32 steps later.
struct RecFlags {
    uint4 f[4];
    __device__ __forceinline__ void fetch(const RecParams &rp, int m2, int n2, int kg, int kblocks, int lane)
    {
        const int kb = kg * 32 + lane;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const bool a = i < 2;
            const int panel = a ? m2 + i : n2 + i - 2;
            f[i] = make_uint4(0, 0, 0, 0);
            if (kb < kblocks && panel < (a ? rp.panels_a : rp.panels_w))
                f[i] = __ldg(reinterpret_cast<const uint4 *>((a ? rp.flags_a : rp.flags_w) + ((int64_t)panel * kblocks + kb) * 16));
        }
    }
    __device__ __forceinline__ uint32_t mask() const           // warp-collective
    {
        uint32_t any = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) any |= f[i].x | f[i].y | f[i].z | f[i].w;
        return __ballot_sync(0xFFFFFFFFu, any != 0);
    }
};

// A step that is not wide brings the scales of its four when it is the first of them or follows a wide step.
__device__ __forceinline__ bool rec_loads_scales(uint32_t wide_mask, int kb)
{
    return (kb & 3) == 0 || ((wide_mask >> ((kb & 31) - 1)) & 1u);
}

template <bool TAIL, bool QOUT>
__global__ void __cluster_dims__(2, 1, 1) __maxnreg__(128)
gemm_rec_kernel(const __grid_constant__ RecMaps tm, const TcParams p, const RecParams rp)
{
    using Cfg = RecCfg;
    constexpr int STAGES = Cfg::STAGES, BN = Cfg::BN;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_gen = smem_raw + (smem_base - ptx::smem_u32(smem_raw));

    const uint32_t zero_base = smem_base + STAGES * Cfg::STAGE_BYTES;
    const uint32_t bar_base = zero_base + Cfg::ZERO_BYTES;
    auto full_bar = [&](int s) { return bar_base + 8u * s; };
    auto empty_bar = [&](int s) { return bar_base + 8u * (STAGES + s); };
    auto tfull_bar = [&](int a) { return bar_base + 8u * (2 * STAGES + a); };
    const uint32_t drained_bar = bar_base + 8u * (2 * STAGES + 2);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem_gen + (bar_base - smem_base) + 8 * (2 * STAGES + 3));
    volatile uint32_t *abort_flag = tmem_slot + 1;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = ptx::cluster_ctarank();         // 0: leader
    const bool leader = rank == 0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            ptx::mbar_init(full_bar(s), 1);
            ptx::mbar_init(empty_bar(s), 1);
        }
        for (int a = 0; a < 2; ++a) ptx::mbar_init(tfull_bar(a), 1);
        ptx::mbar_init(drained_bar, 2 * Cfg::EPI_WARPS);            // the epilogue warps of both CTAs
        *abort_flag = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tm.a);
        ptx::prefetch_tensormap(&tm.w);
        ptx::prefetch_tensormap(&tm.sa);
        ptx::prefetch_tensormap(&tm.sw);
    }
    for (uint32_t i = threadIdx.x; i < Cfg::ZERO_BYTES / 16; i += Cfg::THREADS)
        *reinterpret_cast<uint4 *>(smem_gen + (zero_base - smem_base) + 16 * i) = make_uint4(0, 0, 0, 0);
    ptx::fence_proxy_async_smem();                        // the zeros are read by the MMAs
    if (warp == 1) {
        ptx::tmem_alloc_pair(ptx::smem_u32(tmem_slot), Cfg::TMEM_COLS);
        ptx::tmem_relinquish_pair();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_sync();                                  // the peer's barriers exist before anyone signals them
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    ptx::dep_wait();
    if (threadIdx.x == 0) ptx::dep_trigger();

    const int num_tiles = p.tiles_m * p.tiles_n;          // pair tiles
    const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
    const int kblocks = (p.K + REC_K - 1) / REC_K;
    bool timed_out = false;
    const int kgroups32 = (kblocks + 31) >> 5;

    if (warp == 0 || (warp == 1 && leader)) {
        // both roles walk the tiles in groups of 32 K steps: the warp looks up which of them are wide (the next group's flags
        // are on their way meanwhile), its elected lane issues
        const uint32_t tm_base = __shfl_sync(0xFFFFFFFFu, tmem_base, 0);
        const uint64_t desc_a = smem_desc_rec(smem_base, REC_ROWS * 16), desc_sf = smem_desc_sf_chunk(smem_base);
        bool ready = false;                                   // the next step's operands are there already
        int s = 0;
        uint32_t ph = 0;
        int it = 0;
        uint32_t set = 0;
        RecFlags ahead;
        ahead.fetch(rp, (pair % p.tiles_m) * 2, (pair / p.tiles_m) * 2, 0, kblocks, lane);
        auto load_records = [&](int stage, int m2, int n2, int kb) {                  // this CTA's panel of A and of W
            const uint32_t sa = smem_base + stage * Cfg::STAGE_BYTES, leader_full = ptx::map_to_cta(full_bar(stage), 0);
            ptx::tma_load_2d_pair(sa, &tm.a, 0, ((m2 + (int)rank) * kblocks + kb) * 16, leader_full);
            ptx::tma_load_2d_pair(sa + Cfg::W_OFF, &tm.w, 0, ((n2 + (int)rank) * kblocks + kb) * 16, leader_full);
        };
        // the first stages' records are on their way while the first flags arrive; their bytes are announced, with the
        // scales', in the loop (a barrier's byte count may run ahead of its announcement)
        const int early = pair < num_tiles ? min(STAGES, kblocks) : 0;
        if (warp == 0 && ptx::elect_one())
            for (int kb = 0; kb < early; ++kb) load_records(kb, (pair % p.tiles_m) * 2, (pair / p.tiles_m) * 2, kb);
        for (int t = pair; t < num_tiles; t += npairs, ++it) {
            const int m2 = (t % p.tiles_m) * 2, n2 = (t / p.tiles_m) * 2;            // first panels of the tile
            const int acc = it & 1;
            const uint32_t d_tmem = tm_base + (uint32_t)acc * Cfg::ACC_STEP;
            for (int kg = 0; kg < kgroups32; ++kg) {
                const uint32_t wide_mask = ahead.mask();
                const bool last = kg + 1 == kgroups32;
                const int tn = last ? t + npairs : t;                                // (past the last tile: panels out of range)
                ahead.fetch(rp, (tn % p.tiles_m) * 2, (tn / p.tiles_m) * 2, last ? 0 : kg + 1, kblocks, lane);
                if (timed_out) continue;
                const int kb_end = min(kblocks, 32 * kg + 32);
                if (warp == 0) {
                    const int pa = m2 + (int)rank;
                    for (int kb = 32 * kg; kb < kb_end; ++kb) {
                        if (!__all_sync(0xFFFFFFFFu, ptx::mbar_wait_bounded_relaxed(empty_bar(s), ph ^ 1u, abort_flag, TC_WAIT_LIMIT_NS))) {
                            timed_out = true;
                            break;
                        }
                        if (ptx::elect_one()) {
                            const bool wide = (wide_mask >> (kb & 31)) & 1u;
                            const bool four = rec_loads_scales(wide_mask, kb);
                            const uint32_t bytes = 2 * REC_BYTES + 3 * (wide ? REC_SFW_BYTES : four ? REC_SF_BYTES : 0u);
                            if (leader) ptx::mbar_arrive_expect_tx(full_bar(s), 2 * bytes);
                            const uint32_t leader_full = ptx::map_to_cta(full_bar(s), 0);
                            const uint32_t sa = smem_base + s * Cfg::STAGE_BYTES;
                            if (it > 0 || kb >= early) load_records(s, m2, n2, kb);
                            if (wide) {
                                ptx::tma_load_2d_pair(sa + Cfg::SFA_OFF, &tm.sa_wide, 0, kb * rp.panels_sa + pa, leader_full);
                                ptx::tma_load_2d_pair(sa + Cfg::SFW_OFF, &tm.sw_wide, 0, kb * rp.panels_sw + n2, leader_full);
                            } else if (four) {
                                ptx::tma_load_2d_pair(sa + Cfg::SFA_OFF, &tm.sa, 0, (kb >> 2) * rp.panels_sa + pa, leader_full);
                                ptx::tma_load_2d_pair(sa + Cfg::SFW_OFF, &tm.sw, 0, (kb >> 2) * rp.panels_sw + n2, leader_full);
                            }
                        }
                        if (++s == STAGES) { s = 0; ph ^= 1u; }
                    }
                    continue;
                }
                // tile it may start when the epilogue has left the columns it shares with tile it - 1 (every warp has
                // by then finished tile it - 2, which lay where tile it goes)
                if (kg == 0 && it > 0 &&
                    !__all_sync(0xFFFFFFFFu, ptx::mbar_wait_bounded_relaxed(drained_bar, (uint32_t)(it - 1) & 1u, abort_flag, TC_WAIT_LIMIT_NS))) {
                    timed_out = true;
                    continue;
                }
                ptx::tc_fence_after_sync();
                // One K step; WIDE_MAY: some step of the group is wide.  The common loop is compiled without the wide step: the
                // issuing lane has about 500 clocks per step.
                auto steps = [&](auto may_c) {
                    constexpr bool WIDE_MAY = decltype(may_c)::value;
                    constexpr uint32_t CHUNK = REC_ROWS * 16;                // bytes of one k-chunk of a record
                    for (int kb = 32 * kg; kb < kb_end; ++kb) {
                        if (!ready && !__all_sync(0xFFFFFFFFu, ptx::mbar_wait_bounded(full_bar(s), ph, abort_flag, TC_WAIT_LIMIT_NS))) {
                            timed_out = true;
                            return;
                        }
                        ptx::tc_fence_after_sync();
                        const int cur = s;
                        if (++s == STAGES) { s = 0; ph ^= 1u; }
                        const bool there = ptx::mbar_test(full_bar(s), ph);  // its answer arrives while the MMAs are issued
                        const bool wide = WIDE_MAY && ((wide_mask >> (kb & 31)) & 1u);
                        const bool scales = wide || (WIDE_MAY ? rec_loads_scales(wide_mask, kb) : (kb & 3) == 0);
                        const uint32_t first = set ^ 1u;                     // the set that this step's scales go to, if it loads any
                        if (scales && !wide) set ^= 1u;                      // (a wide step loads twice and ends where it began)
                        if (ptx::elect_one()) {
                            const uint32_t off16 = (uint32_t)cur * (Cfg::STAGE_BYTES >> 4);
                            const uint64_t da = desc_a + off16, dw = da + (Cfg::W_OFF >> 4), dsf = desc_sf + off16;
                            // scales: shared -> tensor memory, executed in order ahead of the MMAs below; `step`: bytes from W's
                            // first panel to its second
                            auto load_scales = [&](uint32_t tsf, uint32_t off, uint32_t step) {
                                tmem_cp_32x128b_warpx4_pair(tsf, dsf + ((Cfg::SFA_OFF + off) >> 4));
                                tmem_cp_32x128b_warpx4_pair(tsf + 4, dsf + ((Cfg::SFW_OFF + off) >> 4));
                                tmem_cp_32x128b_warpx4_pair(tsf + 8, dsf + ((Cfg::SFW_OFF + off + step) >> 4));
                            };
                            if (!wide) {
                                const uint32_t tsf = tm_base + Cfg::SF_COL + set * Cfg::SF_SET;
                                if (scales) load_scales(tsf, 0, REC_SF_BYTES);
                                const uint32_t idesc = idesc_mxf8_e4m3(256, BN, (uint32_t)(kb & 3));
#pragma unroll
                                for (int j = 0; j < REC_K / 32; ++j)
                                    mma_mxf8_ss_pair(d_tmem, da + (uint32_t)(2 * j * CHUNK >> 4), dw + (uint32_t)(2 * j * CHUNK >> 4), idesc, tsf, tsf + 4,
                                                     (kb | j) != 0 ? 1u : 0u);
                            } else {
                                const uint32_t sa = smem_base + cur * Cfg::STAGE_BYTES, sw = sa + Cfg::W_OFF;
#pragma unroll 1
                                for (int h = 0; h < 2; ++h) {
                                    const uint32_t tsf = tm_base + Cfg::SF_COL + (first ^ (uint32_t)h) * Cfg::SF_SET;
                                    load_scales(tsf, 512 * h, REC_SFW_BYTES);
#pragma unroll
                                    for (int j = 0; j < REC_K / 32; ++j) {
                                        const uint32_t ca = sa + (2 * j + h) * CHUNK, cw = sw + (2 * j + h) * CHUNK;
                                        mma_mxf8_ss_pair(d_tmem, smem_desc_rec(ca, zero_base - ca), smem_desc_rec(cw, zero_base - cw),
                                                         idesc_mxf8_e4m3(256, BN, (uint32_t)j), tsf, tsf + 4, (kb | h | j) != 0 ? 1u : 0u);
                                    }
                                }
                            }
                            ptx::mma_commit_pair(empty_bar(cur), 3);         // both CTAs may refill the stage
                        }
                        ready = __all_sync(0xFFFFFFFFu, there);
                    }
                };
                if (wide_mask == 0) steps(std::false_type{});
                else steps(std::true_type{});
                if (kg + 1 == kgroups32 && !timed_out && ptx::elect_one()) ptx::mma_commit_pair(tfull_bar(acc), 3);   // both halves of the accumulator are complete
            }
        }
        __syncwarp();
    } else if (warp >= 2) {
        const int quad = warp & 3;                           // TMEM lane quarter (the hardware's window for this warp)
        const int half = (warp - 2) >> 2;                    // this warp's 128 of the tile's 256 columns
        constexpr int COLS = BN / 2;
        int it = 0;
        for (int t = pair; t < num_tiles && !timed_out; t += npairs, ++it) {
            const int acc = it & 1;
            const uint32_t acc_ph = (uint32_t)(it >> 1) & 1u;
            const int m0 = (t % p.tiles_m) * 256 + (int)rank * 128, n0 = (t / p.tiles_m) * BN;
            const int row = m0 + quad * 32 + lane;
            // the 32 columns shared with the next tile's accumulator come first: the last ones of the first
            // accumulator, the first ones of the second
            const bool down = acc == 0;
            auto column = [&](int i) { return half * COLS + 32 * (down ? COLS / 32 - 1 - i : i); };
            const bool has_shared = down ? half == 1 : half == 0;
            const int rows0 = m0 + quad * 32;
            TailRegs row_ahead;                                     // MXInt result: a row per lane
            FragTail frag_ahead;                                    // fp32 result: the accumulator-fragment shape
            if (TAIL) {                                             // the first chunk's residual: in flight under the MMAs
                if (QOUT) tail_fetch(p, row, n0 + column(0), row_ahead);
                else frag_tail_fetch(p, rows0, n0 + column(0), lane, frag_ahead);
            }
            const bool ok = ptx::mbar_wait_bounded_relaxed(tfull_bar(acc), acc_ph, abort_flag, TC_WAIT_LIMIT_NS);
            if (!__all_sync(0xFFFFFFFFu, ok)) {
                timed_out = true;
                break;
            }
            ptx::tc_fence_after_sync();
            auto release = [&]() {                                  // warp-collective
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive_cluster_relaxed(ptx::map_to_cta(drained_bar, 0));
            };
            if (!has_shared) release();
            const uint32_t t_acc = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)acc * Cfg::ACC_STEP;
#pragma unroll 1
            for (int i = 0; i < COLS / 32; ++i) {
                const int c0 = column(i);
                const int n = n0 + c0;
                if (!QOUT) {
                    uint32_t r[2][16];
                    const FragTail cur = frag_ahead;
                    if (TAIL && i + 1 < COLS / 32) frag_tail_fetch(p, rows0, n0 + column(i + 1), lane, frag_ahead);
                    load_f32_frag(t_acc + (uint32_t)c0, r);
                    if (i == 0 && has_shared) release();
                    frag_store<TAIL>(p, r, cur, rows0, n, lane);
                    continue;
                }
                uint32_t r[32];
                ptx::tmem_ld_32x32(t_acc + (uint32_t)c0, r);
                const TailRegs cur = row_ahead;
                if (TAIL && i + 1 < COLS / 32) tail_fetch(p, row, n0 + column(i + 1), row_ahead);
                ptx::tmem_ld_wait();
                if (i == 0 && has_shared) release();
                if (TAIL) tail_apply(p, cur, n, r);
                store_mxint_chunk(p, row, n, r);
            }
        }
    }

    if (timed_out) {
        *abort_flag = 1;
        atomicOr(p.status, STATUS_TIMEOUT_BIT);
        const uint64_t t0 = ptx::globaltimer_ns();
        while (ptx::globaltimer_ns() - t0 < 100000ull) __nanosleep(1000);
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_sync();          // the peer no longer reads this CTA's shared memory or signals its barriers
    if (warp == 1) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc_pair(tmem_base, Cfg::TMEM_COLS);
    }
}

}  // namespace mx
