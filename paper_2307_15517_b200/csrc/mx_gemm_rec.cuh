// MXInt product on the tensor pipe's block-scaled 8-bit path, CTA pairs (Sec. 3.2: the MXInt dot-product operator
// applies the shared exponent once per block; tcgen05.mma.kind::mxf8f6f4.block_scale is that operator in silicon).
// Operands are records (mx_records.cuh): exact for mantissa widths up to 5 on both sides, blocks of 16 and of 32.
// Products are exact, the 32 products of an MMA step are summed with the scale 2^(Ea+Ew) and accumulate in fp32 in
// tensor memory, as in the bf16 kernels; the 8-bit pipe runs at twice their rate on half their operand bytes.
//
// Two CTAs on neighbouring SMs (a cluster of two) share one 256 x 256 output tile, K step 128: each holds one record
// of A and one of W per step, plus the scales of its own A rows and of all 256 rows of W (the pair's MMA reads the W
// scales from both CTAs' tensor memory).  The warp roles and barriers are those of mx_gemm_tc2.cuh:
//   warp 0      : TMA producer (one lane, in both CTAs; bytes are counted on the leader's barrier)
//   warp 1      : tensor-memory allocation (both CTAs), scale copies and MMA issue (leader only)
//   warps 2..9  : epilogue of the CTA's own 128 rows, two warps per TMEM lane quarter
//
// Tensor memory: 512 columns cannot hold two accumulators of 256 and the scales.  The accumulators overlap by 32
// columns ([0, 256) and [224, 480)), the last 32 columns hold two sets of scales.  The epilogue drains the shared
// columns first and then lets the next tile's MMAs start, so what is exposed between two tiles is one 32-column read.
//
// Wide mode (the flag word equals the call's tag: some row's blocks were too far apart for one scale per record):
// every 32 k take two MMAs, one per half.  The operands' second k-chunk of 16 is then a panel of zeros in
// shared memory -- without swizzle the distance between the two chunks of an MMA is a free field of the descriptor --
// and each half has its own scales.  Twice the MMAs, the rate of the bf16 kernels, exact for any exponents.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "mx_gemm_tc.cuh"
#include "mx_gemm_tc8.cuh"
#include "mx_ptx.cuh"
#include "mx_records.cuh"

namespace mx {

struct RecCfg {
    static constexpr int BN = 256;                        // pair tile: 256 x 256
    static constexpr int STAGES = 5;
    static constexpr uint32_t SFA_OFF = 2 * REC_BYTES;                      // A record, W record, then the scales:
    static constexpr uint32_t SFW_OFF = SFA_OFF + REC_SFW_BYTES;            // own rows of A; both panels of W
    static constexpr uint32_t STAGE_BYTES = SFW_OFF + 2 * REC_SFW_BYTES;    // 35 KB
    static constexpr int EPI_WARPS = 8;
    static constexpr int THREADS = 64 + 32 * EPI_WARPS;
    static constexpr uint32_t EPI_BYTES = EPI_WARPS * 4096;                 // one 32x32 fp32 store buffer per epilogue warp
    static constexpr uint32_t ZERO_BYTES = REC_ROWS * 16;                   // one k-chunk of zeros
    static constexpr uint32_t BAR_BYTES = 256;
    static constexpr uint32_t SMEM_BYTES = STAGES * STAGE_BYTES + EPI_BYTES + ZERO_BYTES + BAR_BYTES + 1024;
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

// Tensor maps over the operands' arrays: records as rows of 1 KB (box: 16 rows = one record), scales as rows of one
// chunk (512 B) or of one record's half-block scales (1 KB), box of one row for A and of two for W.
struct RecMaps { CUtensorMap a, w, sa, sw, sa_wide, sw_wide, y; };

struct RecParams {
    const unsigned long long *flag;          // wide mode when *flag == tag
    unsigned long long tag;
    int panels_sa, panels_sw;                // rows of the scale arrays per K step (group)
};

template <bool TAIL = false>
__global__ void __cluster_dims__(2, 1, 1) __maxnreg__(128)
gemm_rec_kernel(const __grid_constant__ RecMaps tm, const TcParams p, const RecParams rp)
{
    using Cfg = RecCfg;
    constexpr int STAGES = Cfg::STAGES, BN = Cfg::BN;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_gen = smem_raw + (smem_base - ptx::smem_u32(smem_raw));

    const uint32_t epi_base = smem_base + STAGES * Cfg::STAGE_BYTES;
    const uint32_t zero_base = epi_base + Cfg::EPI_BYTES;
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
    auto is_wide = [&]() { return *reinterpret_cast<const volatile unsigned long long *>(rp.flag) == rp.tag; };

    if (warp == 0) {
        if (lane == 0) {
            const bool wide = is_wide();
            int s = 0;
            uint32_t ph = 0;
            for (int t = pair; t < num_tiles && !timed_out; t += npairs) {
                const int pa = (t % p.tiles_m) * 2 + (int)rank;              // this CTA's panel of A and of W
                const int pw0 = (t / p.tiles_m) * 2, pw = pw0 + (int)rank;
                for (int kb = 0; kb < kblocks; ++kb) {
                    if (!ptx::mbar_wait_bounded_cluster(empty_bar(s), ph ^ 1u, abort_flag, TC_WAIT_LIMIT_NS)) {
                        timed_out = true;
                        break;
                    }
                    const bool scales = wide || (kb & 3) == 0;               // this stage brings scales
                    const uint32_t bytes = 2 * REC_BYTES + (scales ? 3 * (wide ? REC_SFW_BYTES : REC_SF_BYTES) : 0u);
                    if (leader) ptx::mbar_arrive_expect_tx(full_bar(s), 2 * bytes);
                    const uint32_t leader_full = ptx::map_to_cta(full_bar(s), 0);
                    const uint32_t sa = smem_base + s * Cfg::STAGE_BYTES;
                    ptx::tma_load_2d_pair(sa, &tm.a, 0, (pa * kblocks + kb) * 16, leader_full);
                    ptx::tma_load_2d_pair(sa + REC_BYTES, &tm.w, 0, (pw * kblocks + kb) * 16, leader_full);
                    if (scales) {
                        const int ks = wide ? kb : kb >> 2;
                        ptx::tma_load_2d_pair(sa + Cfg::SFA_OFF, wide ? &tm.sa_wide : &tm.sa, 0, ks * rp.panels_sa + pa, leader_full);
                        ptx::tma_load_2d_pair(sa + Cfg::SFW_OFF, wide ? &tm.sw_wide : &tm.sw, 0, ks * rp.panels_sw + pw0, leader_full);
                    }
                    if (++s == STAGES) { s = 0; ph ^= 1u; }
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0 && leader) {
            const bool wide = is_wide();
            int s = 0;
            uint32_t ph = 0;
            int it = 0;
            uint32_t set = 0;
            for (int t = pair; t < num_tiles && !timed_out; t += npairs, ++it) {
                const int acc = it & 1;
                // tile it may start when the epilogue has left the columns it shares with tile it - 1 (every warp has
                // by then finished tile it - 2, which lay where tile it goes)
                if (it > 0 && !ptx::mbar_wait_bounded_cluster(drained_bar, (uint32_t)(it - 1) & 1u, abort_flag, TC_WAIT_LIMIT_NS)) {
                    timed_out = true;
                    break;
                }
                ptx::tc_fence_after_sync();
                const uint32_t d_tmem = tmem_base + (uint32_t)acc * Cfg::ACC_STEP;
                for (int kb = 0; kb < kblocks; ++kb) {
                    if (!ptx::mbar_wait_bounded_cluster(full_bar(s), ph, abort_flag, TC_WAIT_LIMIT_NS)) {
                        timed_out = true;
                        break;
                    }
                    ptx::tc_fence_after_sync();
                    const uint32_t sa = smem_base + s * Cfg::STAGE_BYTES;
                    const uint32_t sw = sa + REC_BYTES;
                    constexpr uint32_t CHUNK = REC_ROWS * 16;                // bytes of one k-chunk of a record
                    if (!wide) {
                        if ((kb & 3) == 0) {
                            // four steps' scales: shared -> tensor memory, executed in order ahead of the MMAs below
                            set ^= 1u;
                            const uint32_t tsfa = tmem_base + Cfg::SF_COL + set * Cfg::SF_SET;
                            tmem_cp_32x128b_warpx4_pair(tsfa, smem_desc_sf_chunk(sa + Cfg::SFA_OFF));
                            tmem_cp_32x128b_warpx4_pair(tsfa + 4, smem_desc_sf_chunk(sa + Cfg::SFW_OFF));
                            tmem_cp_32x128b_warpx4_pair(tsfa + 8, smem_desc_sf_chunk(sa + Cfg::SFW_OFF + REC_SF_BYTES));
                        }
                        const uint32_t tsfa = tmem_base + Cfg::SF_COL + set * Cfg::SF_SET;
                        const uint32_t idesc = idesc_mxf8_e4m3(256, BN, (uint32_t)(kb & 3));
#pragma unroll
                        for (int j = 0; j < REC_K / 32; ++j)
                            mma_mxf8_ss_pair(d_tmem, smem_desc_rec(sa + 2 * j * CHUNK, CHUNK), smem_desc_rec(sw + 2 * j * CHUNK, CHUNK),
                                             idesc, tsfa, tsfa + 4, (kb | j) != 0 ? 1u : 0u);
                    } else {
#pragma unroll 1
                        for (int h = 0; h < 2; ++h) {
                            set ^= 1u;
                            const uint32_t tsfa = tmem_base + Cfg::SF_COL + set * Cfg::SF_SET;
                            tmem_cp_32x128b_warpx4_pair(tsfa, smem_desc_sf_chunk(sa + Cfg::SFA_OFF + 512 * h));
                            tmem_cp_32x128b_warpx4_pair(tsfa + 4, smem_desc_sf_chunk(sa + Cfg::SFW_OFF + 512 * h));
                            tmem_cp_32x128b_warpx4_pair(tsfa + 8, smem_desc_sf_chunk(sa + Cfg::SFW_OFF + REC_SFW_BYTES + 512 * h));
#pragma unroll
                            for (int j = 0; j < REC_K / 32; ++j) {
                                const uint32_t ca = sa + (2 * j + h) * CHUNK, cw = sw + (2 * j + h) * CHUNK;
                                mma_mxf8_ss_pair(d_tmem, smem_desc_rec(ca, zero_base - ca), smem_desc_rec(cw, zero_base - cw),
                                                 idesc_mxf8_e4m3(256, BN, (uint32_t)j), tsfa, tsfa + 4, (kb | h | j) != 0 ? 1u : 0u);
                            }
                        }
                    }
                    ptx::mma_commit_pair(empty_bar(s), 3);          // both CTAs may refill the stage
                    if (++s == STAGES) { s = 0; ph ^= 1u; }
                }
                if (timed_out) break;
                ptx::mma_commit_pair(tfull_bar(acc), 3);            // both halves of the accumulator are complete
            }
        }
        __syncwarp();
    } else {
        const int quad = warp & 3;                           // TMEM lane quarter (the hardware's window for this warp)
        const int half = (warp - 2) >> 2;                    // this warp's 128 of the tile's 256 columns
        constexpr int COLS = BN / 2;
        int it = 0;
        uint32_t epi_buf = 0;
        constexpr bool tail = TAIL;
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
            TailRegs ahead;
            if (tail) tail_fetch(p, row, n0 + column(0), ahead);    // the first chunk's residual: in flight under the MMAs
            const bool ok = ptx::mbar_wait_bounded_cluster(tfull_bar(acc), acc_ph, abort_flag, TC_WAIT_LIMIT_NS);
            if (!__all_sync(0xFFFFFFFFu, ok)) {
                timed_out = true;
                break;
            }
            ptx::tc_fence_after_sync();
            auto release = [&]() {                                  // warp-collective
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive_cluster(ptx::map_to_cta(drained_bar, 0));
            };
            if (!has_shared) release();
            const uint32_t t_acc = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)acc * Cfg::ACC_STEP;
#pragma unroll 1
            for (int i = 0; i < COLS / 32; ++i) {
                const int c0 = column(i);
                const int n = n0 + c0;
                if (!tail && p.frag_store) {
                    uint32_t r[2][16];
                    load_f32_frag(t_acc + (uint32_t)c0, r);
                    if (i == 0 && has_shared) release();
                    store_f32_frag_regs(p, r, m0 + quad * 32, n, 0, lane);
                    continue;
                }
                uint32_t r[32];
                ptx::tmem_ld_32x32(t_acc + (uint32_t)c0, r);
                TailRegs cur;
                if (tail) {
                    cur = ahead;                                                          // fetched a chunk ago: has arrived
                    if (i + 1 < COLS / 32) tail_fetch(p, row, n0 + column(i + 1), ahead);  // in flight under this chunk
                }
                ptx::tmem_ld_wait();
                if (i == 0 && has_shared) release();
                if (tail) tail_apply(p, cur, n, r);
                if (p.yq_mant) {
                    store_mxint_chunk(p, row, n, r);
                    continue;
                }
                store_f32_chunk<1>(p, &tm.y, r, row, m0 + quad * 32, n, 0, epi_base + (uint32_t)(warp - 2) * 4096u, epi_buf, lane);
            }
        }
        if (p.tma_store && lane == 0) ptx::bulk_wait_group<0>();
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
