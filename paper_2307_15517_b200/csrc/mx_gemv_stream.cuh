// Decode-shaped MXInt product: a handful of tokens (T <= 16) against weight matrices that are
// streamed from HBM exactly once (Sec. 3.2 MXInt dot-product operator; the paper motivates MX
// formats by the memory footprint of the parameters, Sec. 1 / Sec. 6).
//
// HBM-bound, so the layout of the loads and the number of bytes in flight decide, not the math.
// The math is the literal operator: integer multiply-adds over one block of 32, one shared
// scale per block, blocks added in ascending order in fp32 -- bit-identical to the CUDA-core
// kernel when a row's blocks are not split over warps.
//
//  * weights  : packed 4-bit mantissas [N, K/2] + exponent bytes [N, K/32] (block 32), by coalesced
//               32-bit loads, four blocks and their four exponent bytes per step, two register sets
//               alternating (any address and K; mx_gemv_mma.cuh fetches by TMA where it can).
//  * tokens   : already quantized (int8 or nibble container); each CTA stages them once per
//               layer into shared memory in the operand order of the integer MMA below, together
//               with their float block scales.
//  * per block: a two's-complement nibble moved into the HIGH half of a byte is the signed byte
//               16*q, so one shift/AND pair turns a packed word into the A operand of
//               mma.sync.m16n8k32 (s8 x s8 -> s32) with no sign extension; the accumulator starts
//               at 0x4B400000, so the result register IS the float 1.5*2^23 + 16*P (P = exact
//               integer block sum, |16 P| < 2^22), and two packed FMAs per output pair apply the
//               weight scale (removing the 1.5*2^23) and the token scale (which carries the 1/16).
//
// A warp owns 16 weight rows.  With split > 1 the K range of a row tile is cut into `split`
// contiguous pieces handled by consecutive warps of one CTA and summed in piece order through
// shared memory (deterministic, but no longer the ascending single chain).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "mx_ptx.cuh"
#include "mx_quantize.cuh"

namespace mx {

struct StreamLayer {
    const uint8_t *w_mant;   // [N, K/2] nibbles
    const uint8_t *w_exp;    // [N, K/32]
    const uint8_t *a_mant;   // [T, K] int8 or [T, K/2] nibbles (a_bits <= 4)
    const uint8_t *a_exp;    // [T, K/32]
    const float *bias;       // nullable
    float *y;                // [T, ldy]
    int64_t ldy;
    int N, K, T;
    int a_bits, w_bits;
    int tile_begin;          // index of this layer's first 16-row tile in the launch
    int n_tiles;             // ceil(N / 16)
    // two-row blocks (the paper's (16,2) shape): rows 2i and 2i+1 share row i of the exponent array.  Weights in
    // this form take the register variant of the kernel (the staged exponent boxes assume one row per weight row).
    int w_rows2, a_rows2;    // 0 or 1: shift applied to the row index of w_exp / a_exp
};

struct StreamParams {
    const StreamLayer *layers;   // device memory
    int n_layers;
    int total_tiles;
    int split;                   // 1, 2, 4 or 8
    int max_nb;                  // largest K/32 over the layers (sizes the shared-memory arrays)
    uint32_t *status;            // device status word (bit 0: a bounded wait expired)
    const CUtensorMap *tmaps;    // kernels that load by TMA: two maps per layer (device memory): [2l] over the packed
                                 // mantissas [N, K/2] bytes, box 128 x 16 rows, 128-byte swizzle;
                                 // [2l+1] over the exponent bytes [N, K/32], box 16 x 16 rows
};

// A call of few layers brings its tables along as launch parameters: no copy in front of the kernel.  (A kernel of its own:
// one that chooses between the two at run time reads both through generic pointers, 515 -> 529 us on 2.7 GB of weights.)
constexpr int STREAM_INLINE_LAYERS = 4;
struct StreamInlineParams : StreamParams {
    StreamLayer inline_layers[STREAM_INLINE_LAYERS];
    alignas(64) CUtensorMap inline_maps[2 * STREAM_INLINE_LAYERS];
    __device__ __forceinline__ const StreamLayer *layer_table() const { return inline_layers; }
    __device__ __forceinline__ const CUtensorMap *map_table() const { return inline_maps; }
};
struct StreamTableParams : StreamParams {
    __device__ __forceinline__ const StreamLayer *layer_table() const { return layers; }
    __device__ __forceinline__ const CUtensorMap *map_table() const { return tmaps; }
};

// Register variant, for calls whose tokens leave no room for weight stages in shared memory: 8 warps, each lane prefetches four
// blocks' words with 32-bit loads.
template <int NT> struct StreamCfg {
    static constexpr int WARPS = 8;
    static constexpr int THREADS = WARPS * 32;
    static constexpr int TP = NT * 8;                              // padded token count
    static constexpr size_t tokens_bytes(int max_nb) { return (size_t)max_nb * TP * (32 + 4); }
    static constexpr size_t smem_bytes(int max_nb) { return tokens_bytes(max_nb) + (size_t)WARPS * NT * 4 * 32 * 4; }
};
constexpr uint64_t STREAM_WAIT_LIMIT_NS = 400ull * 1000 * 1000;
constexpr int STREAM_MAGIC_INT = 0x4B400000;        // bit pattern of 1.5 * 2^23
constexpr float STREAM_MAGIC = 12582912.0f;

__device__ __forceinline__ void mma_s8s8_m16n8k32(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                                  uint32_t a3, uint32_t b0, uint32_t b1, const int (&c)[4])
{
    asm volatile(
        "mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%10,%11,%12,%13};"
        : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "r"(c[0]), "r"(c[1]), "r"(c[2]), "r"(c[3]));
}

// NT = number of 8-token column tiles (1: T <= 8, 2: T <= 16).
template <int NT, typename Params>
__global__ void __launch_bounds__(StreamCfg<NT>::THREADS, 1)
gemv_stream_kernel(const __grid_constant__ Params p)
{
    using Cfg = StreamCfg<NT>;
    constexpr int TP = Cfg::TP, WARPS = Cfg::WARPS;
    extern __shared__ __align__(16) uint8_t smem[];
    uint2 *sB = reinterpret_cast<uint2 *>(smem);                 // [nb][TP][4]: (even-k word, odd-k word)
    // [nb][TP] token block scales; they also carry the weights' binary point 2^-(ww-2) and the 1/16
    // of the shifted nibbles, so the weight scale below is the plain 2^(Ew-127)
    float *sCS = reinterpret_cast<float *>(smem + (size_t)p.max_nb * TP * 32);
    float *sRed = sCS + (size_t)p.max_nb * TP;                    // split-K exchange [WARPS][NT][4][32]

    ptx::dep_wait();                          // the quantized tokens come from the previous launch
    if (threadIdx.x == 0) ptx::dep_trigger();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    const int S = p.split, TPR = WARPS / S;                      // row tiles per round of the CTA
    const int per = (p.total_tiles + gridDim.x - 1) / gridDim.x;
    int tile_lo = blockIdx.x * per;
    const int tile_hi = min(tile_lo + per, p.total_tiles);
    const StreamLayer *layers = p.layer_table();
    int li = 0;
    while (li + 1 < p.n_layers && layers[li + 1].tile_begin <= tile_lo) ++li;

    while (tile_lo < tile_hi) {
        const StreamLayer L = layers[li];
        const int l_end = min(tile_hi, L.tile_begin + L.n_tiles);
        const int nb = L.K >> 5;

        // ---- stage this layer's tokens: operand words, block scales, accumulator seeds ----
        __syncthreads();                                         // previous layer fully consumed
        for (int i = threadIdx.x; i < nb * TP * 4; i += Cfg::THREADS) {
            const int tq = i & 3, tok = (i >> 2) % TP, b = (i >> 2) / TP;
            uint32_t lo = 0, hi = 0;                             // 8 mantissas, k = 32b + 8tq ..
            if (tok < L.T) {
                if (L.a_bits <= 4) {
                    const uint32_t pk = __ldg(reinterpret_cast<const uint32_t *>(
                        L.a_mant + (int64_t)tok * (L.K >> 1) + b * 16 + tq * 4));
                    uint32_t by[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) by[j] = (uint32_t)((((int)(pk << (28 - 4 * j))) >> 28) & 0xFF);
                    lo = by[0] | (by[1] << 8) | (by[2] << 16) | (by[3] << 24);
                    hi = by[4] | (by[5] << 8) | (by[6] << 16) | (by[7] << 24);
                } else {
                    const uint2 v = __ldg(reinterpret_cast<const uint2 *>(
                        L.a_mant + (int64_t)tok * L.K + b * 32 + tq * 8));
                    lo = v.x;
                    hi = v.y;
                }
            }
            // MMA slots 4t..4t+3 take the even k of this group of 8, slots 16+4t.. the odd k
            sB[i] = make_uint2(__byte_perm(lo, hi, 0x6420), __byte_perm(lo, hi, 0x7531));
            if (tq == 0) {
                const int eb = tok < L.T ? (int)__ldg(L.a_exp + (int64_t)(tok >> L.a_rows2) * nb + b) : 0;
                // 2^(Ea-127-(wa-2)) * 2^-(ww-2) * 2^-4, every factor an exact power of two
                sCS[b * TP + tok] = f32_scale(eb, L.a_bits) * small_neg_pow2(L.w_bits) * 0.0625f;
            }
        }
        __syncthreads();

        const int64_t w_ld = L.K >> 1;
        for (int base = tile_lo; base < l_end; base += TPR) {
            const int tile = base + warp / S, s = warp % S;
            const bool active = tile < l_end;
            f32x2_t accA[NT], accB[NT];        // rows g / g + 8, tokens (2t, 2t + 1) of each column tile
#pragma unroll
            for (int n = 0; n < NT; ++n) accA[n] = accB[n] = pack2(0.f, 0.f);
            const int r0 = (tile - L.tile_begin) * 16;
            if (active) {
                const int rowA = min(r0 + g, L.N - 1), rowB = min(r0 + g + 8, L.N - 1);
                const uint8_t *mA = L.w_mant + (int64_t)rowA * w_ld + t * 4;
                const uint8_t *mB = L.w_mant + (int64_t)rowB * w_ld + t * 4;
                const uint8_t *eA = L.w_exp + (int64_t)(rowA >> L.w_rows2) * nb;
                const uint8_t *eB = L.w_exp + (int64_t)(rowB >> L.w_rows2) * nb;
                const int b_lo = (nb / S) * s, b_hi = b_lo + nb / S;       // nb % (4*S) == 0
                struct Regs { uint32_t a[4], b[4], ea, eb; };
                // any exponent byte >= 226: 1.5*2^23 * 2^(E-127) is not finite, take two steps there
                auto near_top = [](uint32_t v) {
                    return ((v & 0x80808080u) & ((v & 0x7F7F7F7Fu) + 0x1E1E1E1Eu)) != 0u;
                };
                auto compute_g = [&](int b, const Regs &r, auto top_c) {
                    constexpr bool TOP = decltype(top_c)::value;
                    const f32x2_t neg_magic = pack2(-STREAM_MAGIC, -STREAM_MAGIC);
                    const int seed[4] = {STREAM_MAGIC_INT, STREAM_MAGIC_INT, STREAM_MAGIC_INT, STREAM_MAGIC_INT};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        // weight scale 2^(E-127): exponent byte moved into the float's exponent field
                        // (byte 0 -> the subnormal 2^-127, byte 255 -> Inf, which turns the block into NaN)
                        const uint32_t fa = j == 3 ? (r.ea >> 1) : (r.ea << (23 - 8 * j));
                        const uint32_t fb = j == 3 ? (r.eb >> 1) : (r.eb << (23 - 8 * j));
                        const uint32_t ba = max(fa & 0x7F800000u, 0x00400000u), bb = max(fb & 0x7F800000u, 0x00400000u);
                        const f32x2_t swA = pack2u(ba, ba), swB = pack2u(bb, bb);
                        const f32x2_t mwA = fmul2(swA, neg_magic), mwB = fmul2(swB, neg_magic);
                        // even-k nibbles shifted up, odd-k nibbles already in the high halves: bytes 16*q
                        const uint32_t a0 = (r.a[j] << 4) & 0xF0F0F0F0u, a2 = r.a[j] & 0xF0F0F0F0u;
                        const uint32_t a1 = (r.b[j] << 4) & 0xF0F0F0F0u, a3 = r.b[j] & 0xF0F0F0F0u;
                        const int blk = b + j;
#pragma unroll
                        for (int n = 0; n < NT; ++n) {
                            const uint2 bf = sB[(blk * TP + n * 8 + g) * 4 + t];
                            const f32x2_t sa = *reinterpret_cast<const f32x2_t *>(sCS + blk * TP + n * 8 + 2 * t);
                            int d[4];
                            mma_s8s8_m16n8k32(d, a0, a1, a2, a3, bf.x, bf.y, seed);
                            f32x2_t pA, pB;                       // P * weight scale (rows g, g + 8), exact
                            if (!TOP) {
                                pA = ffma2(pack2u((uint32_t)d[0], (uint32_t)d[1]), swA, mwA);
                                pB = ffma2(pack2u((uint32_t)d[2], (uint32_t)d[3]), swB, mwB);
                            } else {
                                // 1.5*2^23 * scale is not finite up here: subtract first; + 0 * scale keeps
                                // finite results and turns an Inf scale into NaN
                                const float wa_ = __uint_as_float(ba), wb_ = __uint_as_float(bb);
                                pA = pack2(fmaf(0.f, wa_, (__int_as_float(d[0]) - STREAM_MAGIC) * wa_),
                                           fmaf(0.f, wa_, (__int_as_float(d[1]) - STREAM_MAGIC) * wa_));
                                pB = pack2(fmaf(0.f, wb_, (__int_as_float(d[2]) - STREAM_MAGIC) * wb_),
                                           fmaf(0.f, wb_, (__int_as_float(d[3]) - STREAM_MAGIC) * wb_));
                            }
                            accA[n] = ffma2(pA, sa, accA[n]);     // one rounding per block, ascending blocks
                            accB[n] = ffma2(pB, sa, accB[n]);
                        }
                    }
                };
                // The two-step form is needed only when an exponent byte is >= 226.  The decision is taken
                // for the whole warp: the MMA inside is warp-collective and must never run divergent.
                auto compute = [&](int b, const Regs &r) {
                    if (__any_sync(0xFFFFFFFFu, near_top(r.ea | r.eb))) compute_g(b, r, std::true_type{});
                    else compute_g(b, r, std::false_type{});
                };
                auto fetch = [&](int b, Regs &r) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        r.a[j] = __ldcs(reinterpret_cast<const uint32_t *>(mA + (b + j) * 16));
                        r.b[j] = __ldcs(reinterpret_cast<const uint32_t *>(mB + (b + j) * 16));
                    }
                    r.ea = __ldcs(reinterpret_cast<const uint32_t *>(eA + b));
                    r.eb = __ldcs(reinterpret_cast<const uint32_t *>(eB + b));
                };
                // two register sets alternate, so the prefetched words are never copied
                Regs ra, rb;
                fetch(b_lo, ra);
                for (int b = b_lo; b < b_hi; b += 8) {
                    const bool second = b + 4 < b_hi;
                    if (second) fetch(b + 4, rb);
                    compute(b, ra);
                    if (b + 8 < b_hi) fetch(b + 8, ra);
                    if (second) compute(b + 4, rb);
                }
            }
            float acc[NT][4];
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                unpack2(accA[n], acc[n][0], acc[n][1]);
                unpack2(accB[n], acc[n][2], acc[n][3]);
            }
            if (S > 1) {                                             // CTA-uniform branch
                __syncthreads();
#pragma unroll
                for (int n = 0; n < NT; ++n)
#pragma unroll
                    for (int j = 0; j < 4; ++j) sRed[((warp * NT + n) * 4 + j) * 32 + lane] = acc[n][j];
                __syncthreads();
                if (s == 0 && active) {
#pragma unroll
                    for (int n = 0; n < NT; ++n)
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            float v = acc[n][j];
                            for (int q = 1; q < S; ++q) v += sRed[(((warp + q) * NT + n) * 4 + j) * 32 + lane];
                            acc[n][j] = v;
                        }
                }
            }
            if (active && s == 0) {
#pragma unroll
                for (int n = 0; n < NT; ++n)
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int row = r0 + g + (j >> 1) * 8, tok = n * 8 + 2 * t + (j & 1);
                        if (row < L.N && tok < L.T)
                            L.y[(int64_t)tok * L.ldy + row] = L.bias ? acc[n][j] + __ldg(L.bias + row) : acc[n][j];
                    }
            }
        }
        tile_lo = l_end;
        ++li;
    }
}

// ---- one or two tokens ---------------------------------------------------------------------------
// With so few tokens the tensor-core form above is bound by instruction issue: an MMA tile serves eight tokens, and its
// operand set-up and rescale cost the same for one (about 32 warp instructions per 16 x 32 weights).  Here a lane owns a
// weight row: 16 bytes are the 32 mantissas of one block, eight dp4a per token give the exact block sum in one register (the
// same 16 * q bytes, the same 1.5 * 2^23 seed), two fmas apply the scales: about 17 instructions at one token and 5 more for
// the second.  Blocks ascend within a lane, so the result is bit for bit the same chain.
// A warp owns 32 rows and a ring of stages of 32 rows x 16 blocks (four 16-row x 128-byte mantissa boxes, two exponent
// boxes); its loads run on into its next tile and the next layer's while the last ones are consumed.  Tokens are staged once
// per distinct activation tensor, not per layer.  Needs K % 512 == 0 in all layers and 16-byte aligned exponent arrays.
// 2.7 GB of weights, kernel only: 513 -> 471 us at one token (5.2 -> 5.7 TB/s); 0.7 GB: 148 -> 133 us at two; but 147 -> 184
// at three and four, and two MMA row tiles per warp in this frame are slower at any number (eight warps hide less than
// sixteen: 148 -> 214 us at eight tokens), so more tokens stay on the form above.
template <int TOK> struct Stream32Cfg {
    static constexpr int WARPS = 8, THREADS = WARPS * 32, ROWS = 32, CH = 16;
    static constexpr int MANT_BYTES = ROWS * CH * 16;                   // 8 KB
    static constexpr int EXP_BYTES = ROWS * CH;
    static constexpr int STAGE_BYTES = MANT_BYTES + EXP_BYTES;
    static constexpr int MAX_STAGES = 3;
    static constexpr size_t RED_BYTES = (size_t)WARPS * TOK * 32 * 4;      // split-K exchange
    static constexpr size_t smem_bytes(int max_nb, int stages)
    {
        return 1024 + (size_t)WARPS * stages * STAGE_BYTES + RED_BYTES + (size_t)WARPS * MAX_STAGES * 8 + 16 +
               (size_t)max_nb * TOK * (32 + 4);
    }
};

// Any of four exponent bytes from 226 on: 1.5 * 2^23 * 2^(E-127) is not finite, the seed is taken off before the scale.
__device__ __forceinline__ bool stream_near_top(uint32_t v)
{
    return ((v & 0x80808080u) & ((v & 0x7F7F7F7Fu) + 0x1E1E1E1Eu)) != 0u;
}
// Weight scale 2^(E-127) of byte j: moved into the float's exponent field (byte 0 -> the subnormal 2^-127, byte 255 -> Inf,
// which turns the block into NaN).
__device__ __forceinline__ uint32_t stream_scale_bits(uint32_t e4, int j)
{
    return max((j == 3 ? e4 >> 1 : e4 << (23 - 8 * j)) & 0x7F800000u, 0x00400000u);
}

// One stage (16 blocks from `b` on) of 32 rows, a row per lane.
template <int TOK>
__device__ __forceinline__ void dp_step(const uint8_t *mant, const uint8_t *exps, const uint4 *sB, const float *sCS, int b, int lane, float (&acc)[TOK])
{
    const uint8_t *sm = mant + (lane >> 4) * 2048 + (lane & 15) * 128;
    const uint4 ex = *reinterpret_cast<const uint4 *>(exps + lane * 16);
    const uint32_t exw[4] = {ex.x, ex.y, ex.z, ex.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const bool top = stream_near_top(exw[q]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = 4 * q + j;
            const uint4 w = *reinterpret_cast<const uint4 *>(sm + (c >> 3) * 4096 + (((c & 7) ^ (lane & 7)) << 4));
            const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
            const float sw = __uint_as_float(stream_scale_bits(exw[q], j));
            const float mw = sw * -STREAM_MAGIC;
#pragma unroll
            for (int k = 0; k < TOK; ++k) {
                const uint4 t0 = sB[((b + c) * TOK + k) * 2], t1 = sB[((b + c) * TOK + k) * 2 + 1];
                const uint32_t tt[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
                int d = STREAM_MAGIC_INT, d2 = 0;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    d = __dp4a((int)((ww[i] << 4) & 0xF0F0F0F0u), (int)tt[2 * i], d);
                    d2 = __dp4a((int)(ww[i] & 0xF0F0F0F0u), (int)tt[2 * i + 1], d2);
                }
                const float f = __int_as_float(d + d2);                   // 1.5 * 2^23 + 16 P
                float pr;                                                  // P * weight scale, exact
                if (!top) pr = fmaf(f, sw, mw);
                else pr = fmaf(0.f, sw, (f - STREAM_MAGIC) * sw);          // (+ 0 * scale: NaN for an Inf scale)
                acc[k] = fmaf(pr, sCS[(b + c) * TOK + k], acc[k]);         // one rounding per block, ascending blocks
            }
        }
    }
}

template <int TOK, typename Params>
__global__ void __launch_bounds__(Stream32Cfg<TOK>::THREADS, 1)
gemv_stream32_kernel(const __grid_constant__ Params p, int stages, int early)
{
    using Cfg = Stream32Cfg<TOK>;
    constexpr int WARPS = Cfg::WARPS, CH = Cfg::CH, ROWS = Cfg::ROWS;
    extern __shared__ __align__(16) uint8_t smem[];
    uint8_t *sMant = smem + ((1024u - (ptx::smem_u32(smem) & 1023u)) & 1023u);      // [WARPS][stages][MANT_BYTES]
    uint8_t *sExp = sMant + WARPS * stages * Cfg::MANT_BYTES;                         // [WARPS][stages][EXP_BYTES]
    float *sRed = reinterpret_cast<float *>(sExp + WARPS * stages * Cfg::EXP_BYTES);  // split-K exchange
    uint8_t *sBar = reinterpret_cast<uint8_t *>(sRed) + Cfg::RED_BYTES;               // [WARPS][MAX_STAGES] mbarriers
    volatile uint32_t *abort_flag = reinterpret_cast<volatile uint32_t *>(sBar + WARPS * Cfg::MAX_STAGES * 8);
    uint4 *sB = reinterpret_cast<uint4 *>(sBar + WARPS * Cfg::MAX_STAGES * 8 + 16);   // [nb][TOK][2]: per 8 k the even and the odd ones
    float *sCS = reinterpret_cast<float *>(sB + (size_t)p.max_nb * TOK * 2);          // [nb][TOK]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < WARPS * Cfg::MAX_STAGES; ++i) ptx::mbar_init(ptx::smem_u32(sBar) + 8 * i, 1);
        *abort_flag = 0;
        ptx::fence_mbar_init();
    }
    __syncthreads();
    // early: the launch in front is this call's quantizer, which lets this one start only after ITS predecessors are complete
    // and writes tokens only; weights and tables may be read before it has finished
    if (!early) ptx::dep_wait();

    const StreamLayer *layers = p.layer_table();
    const CUtensorMap *tmaps = p.map_table();
    const int S = p.split, TPR = WARPS / S, slot = warp / S, piece = warp % S;
    const int per = (p.total_tiles + gridDim.x - 1) / gridDim.x;
    const int tile_first = blockIdx.x * per, tile_hi = min(tile_first + per, p.total_tiles);
    int li = 0;
    while (li + 1 < p.n_layers && layers[li + 1].tile_begin <= tile_first) ++li;

    // this warp's loads: a cursor over (layer, tile, step) that runs ahead of the arithmetic, across tiles and layers
    const uint32_t my_bar = ptx::smem_u32(sBar) + 8 * warp * Cfg::MAX_STAGES;
    const uint32_t my_mant = ptx::smem_u32(sMant) + warp * stages * Cfg::MANT_BYTES;
    const uint32_t my_exp = ptx::smem_u32(sExp) + warp * stages * Cfg::EXP_BYTES;
    int c_li = li, c_base = tile_first, c_step = 0, c_begin = 0, c_end = 0, c_nsteps = 0, c_b0 = 0, c_stage = 0;
    bool c_live = tile_first < tile_hi;
    auto cursor_layer = [&]() {               // first layer from c_li on that has a tile for this warp
        while (c_live) {
            const StreamLayer &L = layers[c_li];
            c_begin = L.tile_begin;
            c_end = min(tile_hi, L.tile_begin + L.n_tiles);
            if (c_base + slot < c_end) {
                const int nb = L.K >> 5;
                c_nsteps = nb / S / CH;
                c_b0 = nb / S * piece;
                return;
            }
            c_base = c_end;
            ++c_li;
            c_live = c_base < tile_hi;
        }
    };
    auto issue = [&]() {                      // lane 0: the cursor's step into stage c_stage, then one step on
        if (!c_live || *abort_flag != 0) return;
        const uint32_t bar = my_bar + 8 * c_stage, dst = my_mant + c_stage * Cfg::MANT_BYTES, dx = my_exp + c_stage * Cfg::EXP_BYTES;
        const CUtensorMap *tm_m = tmaps + 2 * c_li, *tm_e = tm_m + 1;
        const int r0 = (c_base + slot - c_begin) * ROWS, b = c_b0 + c_step * CH;
        ptx::mbar_arrive_expect_tx(bar, Cfg::STAGE_BYTES);
#pragma unroll
        for (int h = 0; h < 2; ++h) {         // (rows >= N read as zero)
            ptx::tma_load_2d(dst + h * 2048, tm_m, b * 16, r0 + 16 * h, bar);
            ptx::tma_load_2d(dst + (2 + h) * 2048, tm_m, b * 16 + 128, r0 + 16 * h, bar);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) ptx::tma_load_2d(dx + h * 256, tm_e, b, r0 + 16 * h, bar);
        if (++c_stage == stages) c_stage = 0;
        if (++c_step == c_nsteps) {
            c_step = 0;
            c_base += TPR;
            cursor_layer();
        }
    };
    if (lane == 0) {
        cursor_layer();
        for (int i = 0; i < stages; ++i) issue();
    }
    __syncwarp();
    if (early) ptx::dep_wait();               // the quantized tokens
    if (threadIdx.x == 0) ptx::dep_trigger();

    int st = 0;                               // stage and parity of the next step to consume
    uint32_t parity = 0;
    bool timed_out = false;
    const uint8_t *staged = nullptr;          // the activation in shared memory, and the weight width its scales carry
    int staged_bits = 0;
    int tile_lo = tile_first;
    while (tile_lo < tile_hi) {
        const StreamLayer L = layers[li];
        const int l_end = min(tile_hi, L.tile_begin + L.n_tiles);
        const int nb = L.K >> 5;
        if (L.a_mant != staged || L.w_bits != staged_bits) {      // CTA-uniform
            staged = L.a_mant;
            staged_bits = L.w_bits;
            __syncthreads();                  // the previous layer's tokens are consumed
            for (int i = threadIdx.x; i < nb * TOK * 4; i += Cfg::THREADS) {
                const int tq = i & 3, tok = (i >> 2) % TOK, b = (i >> 2) / TOK;
                uint32_t lo = 0, hi = 0;      // 8 mantissas, k = 32b + 8tq ..
                if (tok < L.T) {
                    if (L.a_bits <= 4) {
                        const uint32_t pk = __ldg(reinterpret_cast<const uint32_t *>(L.a_mant + (int64_t)tok * (L.K >> 1) + b * 16 + tq * 4));
                        uint32_t by[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) by[j] = (uint32_t)((((int)(pk << (28 - 4 * j))) >> 28) & 0xFF);
                        lo = by[0] | (by[1] << 8) | (by[2] << 16) | (by[3] << 24);
                        hi = by[4] | (by[5] << 8) | (by[6] << 16) | (by[7] << 24);
                    } else {
                        const uint2 v = __ldg(reinterpret_cast<const uint2 *>(L.a_mant + (int64_t)tok * L.K + b * 32 + tq * 8));
                        lo = v.x;
                        hi = v.y;
                    }
                }
                reinterpret_cast<uint2 *>(sB)[i] = make_uint2(__byte_perm(lo, hi, 0x6420), __byte_perm(lo, hi, 0x7531));
                if (tq == 0) {
                    const int eb = tok < L.T ? (int)__ldg(L.a_exp + (int64_t)(tok >> L.a_rows2) * nb + b) : 0;
                    sCS[b * TOK + tok] = f32_scale(eb, L.a_bits) * small_neg_pow2(L.w_bits) * 0.0625f;
                }
            }
            __syncthreads();
        }
        const int nsteps = nb / S / CH, b_lo = nb / S * piece;
        for (int base = tile_lo; base < l_end; base += TPR) {
            const int tile = base + slot;
            const bool active = tile < l_end;
            float acc[TOK];
#pragma unroll
            for (int k = 0; k < TOK; ++k) acc[k] = 0.f;
            for (int step = 0; active && step < nsteps && !timed_out; ++step) {
                const bool ok = ptx::mbar_wait_bounded(my_bar + 8 * st, parity, abort_flag, STREAM_WAIT_LIMIT_NS);
                if (!__all_sync(0xFFFFFFFFu, ok)) {
                    timed_out = true;
                    *abort_flag = 1;          // the other warps stop issuing as well
                    break;
                }
                const uint8_t *mant = sMant + (warp * stages + st) * Cfg::MANT_BYTES, *exps = sExp + (warp * stages + st) * Cfg::EXP_BYTES;
                dp_step<TOK>(mant, exps, sB, sCS, b_lo + step * CH, lane, acc);
                __syncwarp();                 // every lane is done reading the stage
                if (++st == stages) { st = 0; parity ^= 1u; }
                if (lane == 0) {
                    ptx::fence_proxy_async_smem();
                    issue();
                }
            }
            const int row = (tile - L.tile_begin) * ROWS + lane;
            if (S > 1) {                      // CTA-uniform
                __syncthreads();
#pragma unroll
                for (int k = 0; k < TOK; ++k) sRed[(warp * TOK + k) * 32 + lane] = acc[k];
                __syncthreads();
                if (piece == 0) {
#pragma unroll
                    for (int k = 0; k < TOK; ++k)
                        for (int q = 1; q < S; ++q) acc[k] += sRed[((warp + q) * TOK + k) * 32 + lane];
                }
            }
            if (active && piece == 0 && row < L.N) {
                const float bias = L.bias ? __ldg(L.bias + row) : 0.f;
#pragma unroll
                for (int k = 0; k < TOK; ++k)
                    if (k < L.T) L.y[(int64_t)k * L.ldy + row] = L.bias ? acc[k] + bias : acc[k];
            }
        }
        // (a warp whose wait expired goes through the remaining rounds without steps: the CTA's barriers stay matched)
        tile_lo = l_end;
        ++li;
    }
    if (timed_out) atomicOr(p.status, 1u);
    if (*abort_flag != 0) {                   // copies already in flight get time to land before the shared memory is released
        const uint64_t t0 = ptx::globaltimer_ns();
        while (ptx::globaltimer_ns() - t0 < 100000ull) __nanosleep(1000);
    }
    __syncthreads();
}

}  // namespace mx
