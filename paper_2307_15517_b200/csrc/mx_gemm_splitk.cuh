// Tensor-core MXInt product for few output tiles and long reductions (a short prompt against a narrow projection): the K
// range of every 128 x 128 tile is cut over the CTAs of a cluster.  With a tile per CTA such a call leaves most of the
// chip idle while a few SMs work through all of K (352 x 2048 x 8192: 48 tiles of 128 K steps on 148 SMs).
//
// Operands and arithmetic are those of mx_gemm_tc.cuh (exact bf16, fp32 accumulation in tensor memory).  Every CTA
// accumulates its K steps, leaves its partial tile in its own shared memory (the stage buffers are free by then), and
// after a cluster barrier each CTA adds up the partials of every S-th chunk of 32 columns through distributed shared
// memory, in rank order -- deterministic -- and runs the epilogue on it.  Not persistent: one tile per cluster.
//   warp 0      : TMA producer
//   warp 1      : tensor-memory allocation, MMA issue
//   warps 2..9  : partial tile to shared memory, then reduction and epilogue
// Every mbarrier wait is bounded; a CTA whose wait expired still reaches both cluster barriers.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "mx_gemm_tc.cuh"
#include "mx_ptx.cuh"

namespace mx {

struct SplitKCfg {
    static constexpr int BN = 128;
    static constexpr int STAGES = 6;
    static constexpr uint32_t A_BYTES = TC_BM * TC_BK * 2;
    static constexpr uint32_t STAGE_BYTES = A_BYTES + BN * TC_BK * 2;       // 32 KB
    static constexpr int EPI_WARPS = 8;
    static constexpr int THREADS = 64 + 32 * EPI_WARPS;
    static constexpr uint32_t SMEM_BYTES = STAGES * STAGE_BYTES + 256 + 1024;
    static constexpr uint32_t TMEM_COLS = 128;
    static constexpr int MAX_SPLIT = 4;
};
static_assert(SplitKCfg::STAGES * SplitKCfg::STAGE_BYTES >= TC_BM * SplitKCfg::BN * 4, "the partial tile reuses the stages");

// Offset of the 16-byte group `c4` (of 8) of row `row` in chunk `chunk` of a partial tile; neighbouring rows' groups are
// swizzled so that a row per lane and four rows per warp both read without bank conflicts.
__device__ __forceinline__ uint32_t splitk_offset(int chunk, int row, int c4)
{
    return (uint32_t)(chunk * (TC_BM * 128) + row * 128 + ((c4 ^ (row & 7)) << 4));
}
__device__ __forceinline__ float4 ld_cluster_f32x4(uint32_t cluster_addr)
{
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(cluster_addr) : "memory");
    return v;
}

// The 16-byte groups `c4` of rows row, row + 4, row + 8 and row + 12 of a chunk, added up over the cluster's partial tiles in
// rank order.  Four loads are in flight per CTA of the cluster: a load from another SM takes as long as the rest of a step.
__device__ __forceinline__ void splitk_sum4(uint32_t smem_base, int split, int chunk, int row, int c4, float4 (&v)[4])
{
    for (int s = 0; s < split; ++s) {
        const uint32_t base = ptx::map_to_cta(smem_base, (uint32_t)s);
        float4 x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = ld_cluster_f32x4(base + splitk_offset(chunk, row + 4 * i, c4));
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            v[i].x = s ? v[i].x + x[i].x : x[i].x;
            v[i].y = s ? v[i].y + x[i].y : x[i].y;
            v[i].z = s ? v[i].z + x[i].z : x[i].z;
            v[i].w = s ? v[i].w + x[i].w : x[i].w;
        }
    }
}

// An MXInt result of the 32 rows of lane quarter `quad` (from m0 on) of a chunk (32 columns from n on): the cluster's partials
// added up, a row per lane, so that a block is a lane's own columns.  The sums are taken in whole lines, four rows per warp and
// load, and pass through this CTA's own copy of the chunk, which no other CTA reads: read a row per lane from the other CTAs, a
// request is 16 bytes of 32 lines (352 x 1024 x 1024 with an 8-bit result: the call 19.3 us, now 12.9; 13.3 without a cut).
// Warp-collective, as the next one.
template <bool TAIL>
__device__ __forceinline__ void splitk_chunk_q(const TcParams &p, uint8_t *smem_gen, uint32_t smem_base, int split, int c, int m0, int n,
                                               int quad, int lane)
{
    const int rows0 = m0 + quad * 32;
    if (n >= p.N || rows0 >= p.M) return;                            // warp-uniform
    const int row = rows0 + lane, c4 = lane & 7;
    TailRegs t;
    if (TAIL) tail_fetch(p, row, n, t);
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        const int lr = quad * 32 + 16 * h + (lane >> 3);
        float4 v[4];
        splitk_sum4(smem_base, split, c, lr, c4, v);
#pragma unroll
        for (int i = 0; i < 4; ++i) *reinterpret_cast<float4 *>(smem_gen + splitk_offset(c, lr + 4 * i, c4)) = v[i];
    }
    __syncwarp();
    uint32_t r[32];
#pragma unroll
    for (int v = 0; v < 8; ++v) {
        const uint4 x = *reinterpret_cast<const uint4 *>(smem_gen + splitk_offset(c, quad * 32 + lane, v));
        r[4 * v] = x.x; r[4 * v + 1] = x.y; r[4 * v + 2] = x.z; r[4 * v + 3] = x.w;
    }
    if (TAIL) tail_apply(p, t, n, r);
    store_mxint_chunk(p, row, n, r);
}

// fp32: rows m0 + r4 .. + 4 G - 1 of a chunk, 128 bytes each, all 8 loads of the at most 8 / G partials in flight.
template <bool TAIL, int G>
__device__ __forceinline__ void splitk_rows4(const TcParams &p, uint32_t smem_base, int split, int c, int m0, int n, int r4, int lane)
{
    const int c4 = lane & 7, col = n + 4 * c4, lr = r4 + (lane >> 3);
    if (n >= p.N || m0 + r4 >= p.M) return;                          // warp-uniform
    const float *bias = TAIL ? p.ex_bias : p.bias;
    float4 x[G][8 / G];
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
        for (int s = 0; s < 8 / G; ++s)
            if (s < split) x[g][s] = ld_cluster_f32x4(ptx::map_to_cta(smem_base, (uint32_t)s) + splitk_offset(c, lr + 4 * g, c4));
    const bool vec = col + 4 <= p.N && (p.ldy & 3) == 0 && (reinterpret_cast<uintptr_t>(p.y) & 15) == 0;
    const bool rvec = TAIL && p.residual && col + 4 <= p.N && (p.ldr & 3) == 0 && (reinterpret_cast<uintptr_t>(p.residual) & 15) == 0;
    float b[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) b[k] = bias && col + k < p.N ? __ldg(bias + col + k) : 0.f;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        const int row = m0 + lr + 4 * g;
        float v[4] = {x[g][0].x, x[g][0].y, x[g][0].z, x[g][0].w};
#pragma unroll
        for (int s = 1; s < 8 / G; ++s) {
            if (s < split) { v[0] += x[g][s].x; v[1] += x[g][s].y; v[2] += x[g][s].z; v[3] += x[g][s].w; }
        }
        if (row >= p.M) continue;
        float res[4] = {0.f, 0.f, 0.f, 0.f};
        if (TAIL && p.residual) {
            const float *src = p.residual + (int64_t)row * p.ldr + col;
            if (rvec) {
                const float4 q = __ldg(reinterpret_cast<const float4 *>(src));
                res[0] = q.x; res[1] = q.y; res[2] = q.z; res[3] = q.w;
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (col + k < p.N) res[k] = __ldg(src + k);
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (bias) v[k] += b[k];
            if (TAIL && p.relu) v[k] = v[k] < 0.f ? 0.f : v[k];      // NaN stays NaN
            if (TAIL && p.residual) v[k] += res[k];
        }
        float *dst = p.y + (int64_t)row * p.ldy + col;
        if (vec) {
            *reinterpret_cast<float4 *>(dst) = make_float4(v[0], v[1], v[2], v[3]);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (col + k < p.N) dst[k] = v[k];
        }
    }
}

// The cluster's partial tiles (`chunks` of 32 columns; chunk c is columns 32 (c % row_chunks) from n0 on, rows of panel
// c / row_chunks) added up and written: in units -- MXInt result: the 32 rows of a lane quarter of a chunk; fp32: 4 G of its
// rows -- dealt to all `warps` of all CTAs of the cluster.  A unit's loads from the other SMs take about a microsecond, however
// few they are, so what counts is a warp's number of units: whole chunks dealt to the CTAs (chunk c to CTA c % split, eight
// units one after the other there) left calls of 33..256 rows at 13.4-14.4 us (K x N = 2048 x 2048), 24.4-26.7 (8192 x 2048) and
// 20.2-21.4 (4096 x 4096, up to 128 rows); now 11.7-12.9, 22.5-25.1 and 18.4-19.6.
template <bool TAIL, bool QOUT, int G>
__device__ __forceinline__ void splitk_units(const TcParams &p, uint8_t *smem_gen, uint32_t smem_base, int split, int chunks, int row_chunks,
                                             int m0, int n0, int first, int warps, int lane)
{
    const int per = QOUT ? 4 : 32 / G;
    for (int u = first; u < chunks * per; u += split * warps) {
        const int c = u / per, at = u % per, panel = c / row_chunks, m = m0 + TC_BM * panel, n = n0 + 32 * (c - panel * row_chunks);
        if (QOUT) splitk_chunk_q<TAIL>(p, smem_gen, smem_base, split, c, m, n, at, lane);
        else splitk_rows4<TAIL, G>(p, smem_base, split, c, m, n, 4 * G * at, lane);
    }
}
template <bool TAIL, bool QOUT>
__device__ __forceinline__ void splitk_reduce(const TcParams &p, uint8_t *smem_gen, uint32_t smem_base, int split, int rank, int chunks,
                                              int row_chunks, int m0, int n0, int warp, int warps, int lane)
{
    const int first = rank + split * warp;
    if (QOUT || split > 4) splitk_units<TAIL, QOUT, 1>(p, smem_gen, smem_base, split, chunks, row_chunks, m0, n0, first, warps, lane);
    else if (split > 2) splitk_units<TAIL, false, 2>(p, smem_gen, smem_base, split, chunks, row_chunks, m0, n0, first, warps, lane);
    else splitk_units<TAIL, false, 4>(p, smem_gen, smem_base, split, chunks, row_chunks, m0, n0, first, warps, lane);
}

// QOUT: an MXInt result (yq_mant), else fp32.
template <bool TAIL, bool QOUT>
__global__ void __maxnreg__(128)
gemm_splitk_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_w, const TcParams p, int split)
{
    using Cfg = SplitKCfg;
    constexpr int STAGES = Cfg::STAGES;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_gen = smem_raw + (smem_base - ptx::smem_u32(smem_raw));
    const uint32_t bar_base = smem_base + STAGES * Cfg::STAGE_BYTES;
    auto full_bar = [&](int s) { return bar_base + 8u * s; };
    auto empty_bar = [&](int s) { return bar_base + 8u * (STAGES + s); };
    const uint32_t done_bar = bar_base + 8u * (2 * STAGES);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem_gen + STAGES * Cfg::STAGE_BYTES + 8 * (2 * STAGES + 1));
    volatile uint32_t *abort_flag = tmem_slot + 1;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)ptx::cluster_ctarank(), tile = (int)blockIdx.x / split;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            ptx::mbar_init(full_bar(s), 1);
            ptx::mbar_init(empty_bar(s), 1);
        }
        ptx::mbar_init(done_bar, 1);
        *abort_flag = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tmap_a);
        ptx::prefetch_tensormap(&tmap_w);
    }
    if (warp == 1) {
        ptx::tmem_alloc(ptx::smem_u32(tmem_slot), Cfg::TMEM_COLS);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    ptx::dep_wait();
    if (threadIdx.x == 0) ptx::dep_trigger();

    const int kblocks = (p.K + TC_BK - 1) / TC_BK;                   // split <= kblocks (host): every CTA has a step
    const int kb0 = (int)((int64_t)kblocks * rank / split), kb1 = (int)((int64_t)kblocks * (rank + 1) / split);
    const int m0 = (tile % p.tiles_m) * TC_BM, n0 = (tile / p.tiles_m) * Cfg::BN;
    bool timed_out = false;

    if (warp == 0) {
        int s = 0;
        uint32_t ph = 0;
        for (int kb = kb0; kb < kb1; ++kb) {
            if (!__all_sync(0xFFFFFFFFu, ptx::mbar_wait_bounded(empty_bar(s), ph ^ 1u, abort_flag, TC_WAIT_LIMIT_NS))) {
                timed_out = true;
                break;
            }
            if (ptx::elect_one()) {
                ptx::mbar_arrive_expect_tx(full_bar(s), Cfg::STAGE_BYTES);
                const uint32_t sa = smem_base + s * Cfg::STAGE_BYTES;
                ptx::tma_load_2d(sa, &tmap_a, kb * TC_BK, m0, full_bar(s));
                ptx::tma_load_2d(sa + Cfg::A_BYTES, &tmap_w, kb * TC_BK, n0, full_bar(s));
            }
            if (++s == STAGES) { s = 0; ph ^= 1u; }
        }
        __syncwarp();
    } else if (warp == 1) {
        constexpr uint32_t idesc = ptx::idesc_bf16_f32(TC_BM, Cfg::BN);
        const uint32_t tm = __shfl_sync(0xFFFFFFFFu, tmem_base, 0);
        const uint64_t desc0 = ptx::smem_desc_k_sw128(smem_base, 0);
        int s = 0;
        uint32_t ph = 0;
        bool ready = false;                                          // the next step's operands are there already
        for (int kb = kb0; kb < kb1; ++kb) {
            if (!ready && !__all_sync(0xFFFFFFFFu, ptx::mbar_wait_bounded(full_bar(s), ph, abort_flag, TC_WAIT_LIMIT_NS))) {
                timed_out = true;
                break;
            }
            ptx::tc_fence_after_sync();
            const int cur = s;
            if (++s == STAGES) { s = 0; ph ^= 1u; }
            const bool ahead = ptx::mbar_test(full_bar(s), ph);      // its answer arrives while the MMAs are issued
            if (ptx::elect_one()) {
                const uint64_t da = desc0 + (uint64_t)((uint32_t)cur * (Cfg::STAGE_BYTES >> 4)), dw = da + (Cfg::A_BYTES >> 4);
#pragma unroll
                for (int j = 0; j < TC_BK / 16; ++j) ptx::mma_bf16_ss(tm, da + 2u * j, dw + 2u * j, idesc, (kb != kb0 || j != 0) ? 1u : 0u);
                ptx::mma_commit(empty_bar(cur));
            }
            ready = __all_sync(0xFFFFFFFFu, ahead);
        }
        if (!timed_out && ptx::elect_one()) ptx::mma_commit(done_bar);
        __syncwarp();
    } else {
        // the partial tile: tensor memory -> this CTA's shared memory.  All its loads have landed and all its MMAs have
        // read them when done_bar completes.
        const int quad = warp & 3, half = (warp - 2) >> 2;
        const bool ok = ptx::mbar_wait_bounded(done_bar, 0, abort_flag, TC_WAIT_LIMIT_NS);
        if (__all_sync(0xFFFFFFFFu, ok)) {
            ptx::tc_fence_after_sync();
            const int row = quad * 32 + lane;
#pragma unroll 1
            for (int c = 2 * half; c < 2 * half + 2; ++c) {
                uint32_t r[32];
                ptx::tmem_ld_32x32(tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(32 * c), r);
                ptx::tmem_ld_wait();
#pragma unroll
                for (int v = 0; v < 8; ++v)
                    *reinterpret_cast<uint4 *>(smem_gen + splitk_offset(c, row, v)) = make_uint4(r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
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
    ptx::cluster_sync();                                             // every partial tile is in place

    if (warp >= 2)
        splitk_reduce<TAIL, QOUT>(p, smem_gen, smem_base, split, rank, Cfg::BN / 32, Cfg::BN / 32, m0, n0, warp - 2, Cfg::EPI_WARPS, lane);
    __syncwarp();
    ptx::tc_fence_before_sync();
    ptx::cluster_sync();                                             // nobody reads this CTA's partial tile any more
    if (warp == 1) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(tmem_base, Cfg::TMEM_COLS);
    }
}

}  // namespace mx
