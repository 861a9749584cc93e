// The bf16 product on CTA pairs with wide tiles: 256 x W, W a multiple of 32 up to 512 that the host picks so that the tiles
// fill whole waves of the chip's pairs (Sec. 3.2 operator on exactly decoded operands, as mx_gemm_tc2.cuh).
//
// Both halves of a tile's columns are MMAs of their own (N = W / 2) on the same rows of A, which are fetched once: per K step
// of 64 a pair moves (256 + W) * 128 bytes for 256 * W * 64 products, a quarter less than 256 x 256 tiles at W = 512 -- an SM
// takes in 58 bytes per clock and needs 64 for those at the pipe's rate.  The accumulator takes W of the 512 columns of tensor
// memory, so there is one: the next tile's MMAs start when the epilogue has drained it (its operands are staged by then).
// What it gives is the choice of a width that fills whole rounds (wide_pair_tile): 512 x 11008 x 4096 61 -> 45 us for the product,
// 2048 x 4096 x 16384 177 -> 165 (1.67 PFLOP/s), bound by the tensor pipe under the power cap.  Same bits as the pair kernel.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "mx_gemm_rec.cuh"
#include "mx_gemm_tc.cuh"
#include "mx_ptx.cuh"

namespace mx {

struct TcwCfg {
    static constexpr int MAX_W = 512, MAX_STAGES = 8;
    static constexpr uint32_t A_BYTES = TC_BM * TC_BK * 2;          // this CTA's 128 rows of A
    static constexpr int EPI_WARPS = 8;
    static constexpr int THREADS = 64 + 32 * EPI_WARPS;
    static constexpr uint32_t BAR_BYTES = 256;
    static constexpr uint32_t TMEM_COLS = 512;
    static constexpr uint32_t stage_bytes(int w) { return A_BYTES + (uint32_t)w * (TC_BK * 2) / 2; }      // ... and W / 2 rows of W
    static constexpr uint32_t smem_bytes(int w, int stages) { return stages * stage_bytes(w) + BAR_BYTES + 1024; }
};

template <bool TAIL, bool QOUT>
__global__ void __cluster_dims__(2, 1, 1) __maxnreg__(128)
gemm_tcw_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_w, const TcParams p,
                const int width, const int stages)
{
    using Cfg = TcwCfg;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_gen = smem_raw + (smem_base - ptx::smem_u32(smem_raw));
    const uint32_t stage_bytes = Cfg::stage_bytes(width);
    const uint32_t bar_base = smem_base + stages * stage_bytes;
    auto full_bar = [&](int s) { return bar_base + 8u * s; };
    auto empty_bar = [&](int s) { return bar_base + 8u * (Cfg::MAX_STAGES + s); };
    const uint32_t tfull_bar = bar_base + 8u * (2 * Cfg::MAX_STAGES), tempty_bar = tfull_bar + 8u;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem_gen + stages * stage_bytes + 8 * (2 * Cfg::MAX_STAGES + 2));
    volatile uint32_t *abort_flag = tmem_slot + 1;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = ptx::cluster_ctarank();         // 0: leader
    const bool leader = rank == 0;
    const int bn = width >> 1;                            // N of one MMA

    if (threadIdx.x == 0) {
        for (int s = 0; s < Cfg::MAX_STAGES; ++s) {
            ptx::mbar_init(full_bar(s), 1);
            ptx::mbar_init(empty_bar(s), 1);
        }
        ptx::mbar_init(tfull_bar, 1);
        ptx::mbar_init(tempty_bar, 2 * Cfg::EPI_WARPS);   // the epilogue warps of both CTAs
        *abort_flag = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tmap_a);
        ptx::prefetch_tensormap(&tmap_w);
    }
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

    const int num_tiles = p.tiles_m * p.tiles_n;
    const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
    const int kblocks = (p.K + TC_BK - 1) / TC_BK;
    bool timed_out = false;

    if (warp == 0) {
        int s = 0;
        uint32_t ph = 0;
        for (int t = pair; t < num_tiles && !timed_out; t += npairs) {
            const int m0 = (t % p.tiles_m) * 256 + (int)rank * 128;
            const int n0 = (t / p.tiles_m) * width + (int)rank * (bn / 2);     // this CTA's rows of either half
            for (int kb = 0; kb < kblocks; ++kb) {
                if (!__all_sync(0xFFFFFFFFu, ptx::mbar_wait_bounded_relaxed(empty_bar(s), ph ^ 1u, abort_flag, TC_WAIT_LIMIT_NS))) {
                    timed_out = true;
                    break;
                }
                if (ptx::elect_one()) {
                    if (leader) ptx::mbar_arrive_expect_tx(full_bar(s), 2 * stage_bytes);
                    const uint32_t leader_full = ptx::map_to_cta(full_bar(s), 0);
                    const uint32_t sa = smem_base + s * stage_bytes, sw = sa + Cfg::A_BYTES;
                    ptx::tma_load_2d_pair(sa, &tmap_a, kb * TC_BK, m0, leader_full);
                    ptx::tma_load_2d_pair(sw, &tmap_w, kb * TC_BK, n0, leader_full);
                    ptx::tma_load_2d_pair(sw + (uint32_t)bn * TC_BK, &tmap_w, kb * TC_BK, n0 + bn, leader_full);
                }
                if (++s == stages) { s = 0; ph ^= 1u; }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        const uint32_t idesc = ptx::idesc_bf16_f32(256, bn);
        const uint32_t tm = __shfl_sync(0xFFFFFFFFu, tmem_base, 0);
        const uint64_t desc0 = ptx::smem_desc_k_sw128(smem_base, 0);
        const uint32_t half16 = (uint32_t)bn * TC_BK >> 4;       // a half's rows, in units of 16 bytes
        int s = 0, it = 0;
        uint32_t ph = 0;
        bool ready = false;                                      // the next step's operands are there already
        for (int t = leader ? pair : num_tiles; t < num_tiles && !timed_out; t += npairs, ++it) {
            bool ok = ptx::mbar_wait_bounded_relaxed(tempty_bar, ((uint32_t)it & 1u) ^ 1u, abort_flag, TC_WAIT_LIMIT_NS);
            for (int kb = 0; kb < kblocks; ++kb) {
                if (kb == 0 || !ready) {
                    ok = ok && (ready || ptx::mbar_wait_bounded(full_bar(s), ph, abort_flag, TC_WAIT_LIMIT_NS));
                    if (!__all_sync(0xFFFFFFFFu, ok)) {
                        timed_out = true;
                        break;
                    }
                }
                ptx::tc_fence_after_sync();
                const int cur = s;
                if (++s == stages) { s = 0; ph ^= 1u; }
                const bool ahead = ptx::mbar_test(full_bar(s), ph);      // its answer arrives while the MMAs are issued
                if (ptx::elect_one()) {
                    const uint64_t da = desc0 + (uint64_t)((uint32_t)cur * (stage_bytes >> 4)), dw = da + (Cfg::A_BYTES >> 4);
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int j = 0; j < TC_BK / 16; ++j)
                            ptx::mma_bf16_ss_pair(tm + (uint32_t)(h * bn), da + 2u * j, dw + (h ? half16 : 0u) + 2u * j, idesc, (kb | j) != 0 ? 1u : 0u);
                    ptx::mma_commit_pair(empty_bar(cur), 3);             // both CTAs may refill the stage
                }
                ready = __all_sync(0xFFFFFFFFu, ahead);
            }
            if (timed_out) break;
            if (ptx::elect_one()) ptx::mma_commit_pair(tfull_bar, 3);
        }
        __syncwarp();
    } else {
        const int quad = warp & 3;                           // TMEM lane quarter (the hardware's window for this warp)
        const int group = (warp - 2) >> 2;                   // even or odd chunks of 32 columns
        int it = 0;
        for (int t = pair; t < num_tiles && !timed_out; t += npairs, ++it) {
            const int m0 = (t % p.tiles_m) * 256 + (int)rank * 128, n0 = (t / p.tiles_m) * width;
            const int rows0 = m0 + quad * 32, row = rows0 + lane;
            TailRegs row_ahead;                              // MXInt result: a row per lane
            FragTail frag_ahead;                             // fp32 result: the accumulator-fragment shape
            if (TAIL) {                                      // the first chunk's residual: in flight under the MMAs
                if (QOUT) tail_fetch(p, row, n0 + 32 * group, row_ahead);
                else frag_tail_fetch(p, rows0, n0 + 32 * group, lane, frag_ahead);
            }
            const bool ok = ptx::mbar_wait_bounded_relaxed(tfull_bar, (uint32_t)it & 1u, abort_flag, TC_WAIT_LIMIT_NS);
            if (!__all_sync(0xFFFFFFFFu, ok)) {
                timed_out = true;
                break;
            }
            ptx::tc_fence_after_sync();
            const uint32_t t_acc = tmem_base + ((uint32_t)(quad * 32) << 16);
#pragma unroll 1
            for (int c0 = 32 * group; c0 < width; c0 += 64) {
                const int n = n0 + c0;
                if (!QOUT) {
                    uint32_t r[2][16];
                    const FragTail cur = frag_ahead;
                    if (TAIL && c0 + 64 < width) frag_tail_fetch(p, rows0, n + 64, lane, frag_ahead);
                    load_f32_frag(t_acc + (uint32_t)c0, r);
                    frag_store<TAIL>(p, r, cur, rows0, n, lane);
                    continue;
                }
                uint32_t r[32];
                ptx::tmem_ld_32x32(t_acc + (uint32_t)c0, r);
                const TailRegs cur = row_ahead;
                if (TAIL && c0 + 64 < width) tail_fetch(p, row, n + 64, row_ahead);
                ptx::tmem_ld_wait();
                if (TAIL) tail_apply(p, cur, n, r);
                store_mxint_chunk(p, row, n, r);
            }
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive_cluster_relaxed(ptx::map_to_cta(tempty_bar, 0));
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
