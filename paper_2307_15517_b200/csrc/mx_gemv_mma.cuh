// Decode-shaped MXInt products on the integer tensor pipe of the SM (Sec. 3.2 dot-product operator): few tokens against packed
// weights that are read once.
//
//   gemv_mma_kernel    : many layers in one launch (mx_linear_grouped, up to 16 tokens), tokens quantized by a launch in front
//   gemv_single_kernel : one layer in one launch (mx_linear, up to 32), tokens quantized here, K cut over a thread-block cluster
//
// Both share the step below: a warp owns 16 weight rows and takes 256 bytes of each per step, staged by two tiled TMA loads
// of 16 rows x 128 bytes (issued back to back, so that DRAM sees 256 contiguous bytes of a row) and read back with ldmatrix:
// one instruction hands lane (g, t) = (lane / 4, lane % 4) word t of four 16-byte chunks of row g.
//   * 4-bit weights: a two's-complement nibble moved into the HIGH half of a byte is the signed byte 16 q, so a shift and two
//     ANDs turn a word into the even- and the odd-k operand registers of mma.m16n8k32 (s8 x s8 -> s32); tokens are staged in
//     the same order.  8-bit weights are the operand registers as they are.
//   * blocks of 16: 8-bit weights take mma.m16n8k16; 4-bit ones take mma.m16n8k32 twice, with the tokens of the other block
//     masked to zero (lanes t = 0, 1 of a word hold the first block, t = 2, 3 the second).
//   * the accumulator starts at 0x4B400000, so the result register IS the float 1.5 * 2^23 + P (P = the exact block sum,
//     |P| < 2^22); a packed fma removes the 1.5 * 2^23 and applies the weight scale, a second one applies the token scale and
//     adds: one fp32 rounding per block, blocks ascending -- the bits of the CUDA-core kernel where K is not cut.
//   * the packed fma wants exponent bytes in 1 .. 225 (2^E * 1.5 * 2^23 finite, 2^E normal): one vote per step looks at all
//     of them; steps with others take the two-step form.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "mx_gemv_stream.cuh"
#include "mx_ptx.cuh"
#include "mx_quantize.cuh"

namespace mx {

template <int NT, bool NIB, int BLOCK> struct MmaStep {
    static constexpr int TP = 8 * NT;                              // tokens, padded to column tiles of the MMA
    static constexpr int KGROUP = NIB ? 128 : 64;                  // k of 64 mantissa bytes: four 16-byte chunks of a row
    static constexpr int GROUPS = 4;                               // groups per step
    static constexpr int KU = KGROUP / 32;                         // MMAs of 32 k per group
    static constexpr int PER = 32 / BLOCK;                         // blocks per 32 k
    static constexpr int GB = KGROUP / BLOCK;                      // blocks = exponent bytes of a row per group: 4, 8, 2, 4
    static constexpr int MANT_BYTES = 4096;                        // 16 rows x 256 bytes
    static constexpr int EXP_BYTES = 16 * GROUPS * GB;
    // staged tokens, column tiles in pairs (P = min(NT, 2)): operand words per group [KU][NT / P][32 lanes][P] uint2, then over
    // all groups the block scales [GB][NT / P][4][P] float2
    static constexpr int B_GROUP = KU * 32 * NT;                   // uint2
    static constexpr int S_GROUP = GB * 4 * NT;                    // float2
    static constexpr size_t token_bytes(int groups) { return (size_t)groups * (B_GROUP + S_GROUP) * 8; }
};

__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_s8s8_m16n8k16(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0, const int (&c)[4])
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%7,%8,%9,%10};"
                 : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
                 : "r"(a0), "r"(a1), "r"(b0), "r"(c[0]), "r"(c[1]), "r"(c[2]), "r"(c[3]));
}
// 4 bytes global -> shared in the background; the bytes from `valid` on are written as zeros.
__device__ __forceinline__ void cp_async4(uint32_t dst, const void *src, int valid)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(valid) : "memory");
}
__device__ __forceinline__ void cp_async8(uint32_t dst, const void *src, int valid)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(valid) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// Arrives on `bar` when this thread's copies so far are in shared memory (one of the barrier's expected arrivals).
__device__ __forceinline__ void cp_async_arrive(uint32_t bar)
{
    asm volatile("cp.async.mbarrier.arrive.noinc.shared.b64 [%0];" ::"r"(bar) : "memory");
}

// Any byte of the word 0 or >= 226: the exponent bytes that the one-step rescale does not take.
__device__ __forceinline__ bool exps_rare(uint32_t v)
{
    return stream_near_top(v) || ((v - 0x01010101u) & ~v & 0x80808080u) != 0u;
}

// 2^64 times a token scale, as a finite number (where that overflows the term does, unless its mantissas are zero).
__device__ __forceinline__ float stream_scale_up(float s)
{
    const float u = s * 0x1p64f;
    return u == INFINITY ? 0x1p127f : u;
}

// One group: the four words of this lane for rows g and g + 8, their exponent bytes, the group's tokens.
template <int NT, bool NIB, int BLOCK, bool RARE>
__device__ __forceinline__ void mma_group(const uint32_t (&wa)[4], const uint32_t (&wb)[4], const uint32_t *ea, const uint32_t *eb,
                                          const uint2 *sB, const f32x2_t *sCS, int lane, f32x2_t (&accA)[NT], f32x2_t (&accB)[NT])
{
    using G = MmaStep<NT, NIB, BLOCK>;
    const f32x2_t neg_magic = pack2(-STREAM_MAGIC, -STREAM_MAGIC);
    const int seed[4] = {STREAM_MAGIC_INT, STREAM_MAGIC_INT, STREAM_MAGIC_INT, STREAM_MAGIC_INT};
    const int t = lane & 3;
#pragma unroll
    for (int u = 0; u < G::KU; ++u) {
        // tokens in pairs of column tiles: 16-byte loads of the operand words and of the scales
        uint32_t bf[NT][2];
        if (NT == 1) {
            const uint2 v = sB[u * 32 + lane];
            bf[0][0] = v.x; bf[0][1] = v.y;
        } else {
#pragma unroll
            for (int n = 0; n < NT; n += 2) {
                const uint4 v = reinterpret_cast<const uint4 *>(sB)[(u * (NT / 2) + n / 2) * 32 + lane];
                bf[n][0] = v.x; bf[n][1] = v.y; bf[(n + 1) % NT][0] = v.z; bf[(n + 1) % NT][1] = v.w;
            }
        }
        uint32_t a0, a1, a2, a3;
        if (NIB) {
            a0 = (wa[u] << 4) & 0xF0F0F0F0u; a2 = wa[u] & 0xF0F0F0F0u;
            a1 = (wb[u] << 4) & 0xF0F0F0F0u; a3 = wb[u] & 0xF0F0F0F0u;
        } else {
            a0 = wa[2 * u % 4]; a1 = wb[2 * u % 4]; a2 = wa[(2 * u + 1) % 4]; a3 = wb[(2 * u + 1) % 4];
        }
#pragma unroll
        for (int h = 0; h < G::PER; ++h) {
            const int blk = u * G::PER + h;
            const uint32_t xa = ea[blk >> 2], xb = eb[blk >> 2];
            uint32_t ba, bb;
            if (RARE) {
                ba = stream_scale_bits(xa, blk & 3); bb = stream_scale_bits(xb, blk & 3);
            } else {
                ba = ((blk & 3) == 3 ? xa >> 1 : xa << (23 - 8 * (blk & 3))) & 0x7F800000u;
                bb = ((blk & 3) == 3 ? xb >> 1 : xb << (23 - 8 * (blk & 3))) & 0x7F800000u;
            }
            const f32x2_t swA = pack2u(ba, ba), swB = pack2u(bb, bb);
            const f32x2_t mwA = fmul2(swA, neg_magic), mwB = fmul2(swB, neg_magic);
            // all column tiles' MMAs first, then their rescales: the warp has NT chains in flight
            int dd[NT][4];
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                const uint32_t b0 = bf[n][0], b1 = bf[n][1];
                if (BLOCK == 32) {
                    mma_s8s8_m16n8k32(dd[n], a0, a1, a2, a3, b0, b1, seed);
                } else if (NIB) {
                    const bool mine = (t >> 1) == h;
                    mma_s8s8_m16n8k32(dd[n], a0, a1, a2, a3, mine ? b0 : 0u, mine ? b1 : 0u, seed);
                } else {
                    mma_s8s8_m16n8k16(dd[n], h ? a2 : a0, h ? a3 : a1, h ? b1 : b0, seed);
                }
            }
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                f32x2_t sa;
                if (NT == 1) {
                    sa = sCS[blk * 4 + t];
                } else {
                    const ulonglong2 w = reinterpret_cast<const ulonglong2 *>(sCS)[(blk * (NT / 2) + n / 2) * 4 + t];
                    sa = n & 1 ? w.y : w.x;
                }
                const int (&d)[4] = dd[n];
                f32x2_t pA, pB;                       // P * weight scale (rows g, g + 8), exact
                if (!RARE) {
                    pA = ffma2(pack2u((uint32_t)d[0], (uint32_t)d[1]), swA, mwA);
                    pB = ffma2(pack2u((uint32_t)d[2], (uint32_t)d[3]), swB, mwB);
                } else {
                    // the seed first; + 0 * scale turns an infinite scale into NaN.  Near the top of the range 2^64 changes sides,
                    // so that P * weight scale stays finite where the term does
                    const bool ta = ba >= 226u << 23, tb = bb >= 226u << 23;
                    const float fa = __uint_as_float(ba) * (ta ? 0x1p-64f : 1.f), fb = __uint_as_float(bb) * (tb ? 0x1p-64f : 1.f);
                    pA = pack2(fmaf(0.f, fa, (__int_as_float(d[0]) - STREAM_MAGIC) * fa),
                               fmaf(0.f, fa, (__int_as_float(d[1]) - STREAM_MAGIC) * fa));
                    pB = pack2(fmaf(0.f, fb, (__int_as_float(d[2]) - STREAM_MAGIC) * fb),
                               fmaf(0.f, fb, (__int_as_float(d[3]) - STREAM_MAGIC) * fb));
                    float s0, s1;
                    unpack2(sa, s0, s1);
                    const f32x2_t up = pack2(stream_scale_up(s0), stream_scale_up(s1));
                    accA[n] = ffma2(pA, ta ? up : sa, accA[n]);
                    accB[n] = ffma2(pB, tb ? up : sa, accB[n]);
                    continue;
                }
                accA[n] = ffma2(pA, sa, accA[n]);     // one rounding per block, ascending blocks
                accB[n] = ffma2(pB, sa, accB[n]);
            }
        }
    }
}

// One staged step of up to four groups.  mant, exps: the stage (shared); sB, sCS: the tokens of the step's first group.
template <int NT, bool NIB, int BLOCK>
__device__ __forceinline__ void mma_step(uint32_t mant, const uint8_t *exps, const uint2 *sB, const f32x2_t *sCS, int groups,
                                         int lane, f32x2_t (&accA)[NT], f32x2_t (&accB)[NT])
{
    using G = MmaStep<NT, NIB, BLOCK>;
    constexpr int EW = (G::GB + 3) / 4;                       // exponent words per group
    const int g = lane >> 2, t = lane & 3;
    // 16-byte chunk c of row r of a box lies at chunk c ^ (r & 7): lane l addresses row l % 8 of chunk 4 * (group % 2) + l / 8
    const uint32_t swz0 = (uint32_t)((lane & 7) * 128 + (((lane >> 3) ^ (lane & 7)) << 4)), swz1 = swz0 ^ 64u;
    const uint8_t *xa = exps + g * (4 * G::GB), *xb = xa + 8 * (4 * G::GB);
    bool rare;                                                // every lane looks at a quarter of its rows' bytes
    if (G::GB == 2) {
        const uint32_t v = (uint32_t)*reinterpret_cast<const uint16_t *>(xa + 2 * t) |
                           ((uint32_t)*reinterpret_cast<const uint16_t *>(xb + 2 * t) << 16);
        rare = exps_rare(v);
    } else {
        rare = false;
#pragma unroll
        for (int w = 0; w < EW; ++w)
            rare |= exps_rare(*reinterpret_cast<const uint32_t *>(xa + G::GB * t + 4 * w)) ||
                    exps_rare(*reinterpret_cast<const uint32_t *>(xb + G::GB * t + 4 * w));
    }
    rare = rare && t < groups;
    auto one = [&](int q, auto rare_c) {
        uint32_t wa[4], wb[4], ea[EW], eb[EW];
        const uint32_t at = mant + (uint32_t)(q >> 1) * 2048u + ((q & 1) ? swz1 : swz0);
        ldmatrix_x4(at, wa);
        ldmatrix_x4(at + 1024u, wb);
        if (G::GB == 2) {
            ea[0] = *reinterpret_cast<const uint16_t *>(xa + 2 * q);
            eb[0] = *reinterpret_cast<const uint16_t *>(xb + 2 * q);
        } else {
#pragma unroll
            for (int w = 0; w < EW; ++w) {
                ea[w] = *reinterpret_cast<const uint32_t *>(xa + G::GB * q + 4 * w);
                eb[w] = *reinterpret_cast<const uint32_t *>(xb + G::GB * q + 4 * w);
            }
        }
        mma_group<NT, NIB, BLOCK, decltype(rare_c)::value>(wa, wb, ea, eb, sB + q * G::B_GROUP, sCS + q * G::S_GROUP, lane, accA, accB);
    };
    // the MMA is warp-collective: the form is chosen for the whole warp, the number of groups is warp-uniform
    if (!__any_sync(0xFFFFFFFFu, rare)) {
#pragma unroll
        for (int q = 0; q < G::GROUPS; ++q) {
            if (q >= groups) break;
            one(q, std::false_type{});
        }
    } else {
#pragma unroll 1
        for (int q = 0; q < groups; ++q) one(q, std::true_type{});
    }
}

// Position of token `tok`'s block scale (float index) and of its eight mantissas k = 32 u + 8 tq .. + 7 in the staged tokens.
template <int NT> __device__ __forceinline__ int token_scale_at(int blk, int tok)
{
    constexpr int P = NT < 2 ? 1 : 2;
    const int n = tok >> 3;
    return (((blk * (NT / P) + n / P) * 4 + ((tok & 7) >> 1)) * P + n % P) * 2 + (tok & 1);
}
template <int NT, bool NIB> __device__ __forceinline__ void put_token_words(uint2 *sB, int u, int tok, int tq, uint32_t lo, uint32_t hi)
{
    constexpr int P = NT < 2 ? 1 : 2;
    const int g = tok & 7, n = tok >> 3, base = (u * (NT / P) + n / P) * 32 + g * 4;      // lane g * 4 + t holds column g's slots
    if (NIB) {            // MMA slots 4t..4t+3 take the even k of this group of 8, slots 16+4t.. the odd k
        sB[(base + tq) * P + n % P] = make_uint2(__byte_perm(lo, hi, 0x6420), __byte_perm(lo, hi, 0x7531));
    } else {              // words 2 tq, 2 tq + 1 of 32 bytes: first register of lanes t = 0..3, then the second
        uint32_t *w = reinterpret_cast<uint32_t *>(sB);
        const int t0 = (2 * tq) & 3, r = tq >> 1;
        w[((base + t0) * P + n % P) * 2 + r] = lo;
        w[((base + t0 + 1) * P + n % P) * 2 + r] = hi;
    }
}

// ---- many layers, tokens quantized beforehand ------------------------------------------------------
// Persistent: a CTA owns a contiguous range of the launch's 16-row tiles, warp w of it every TPR-th; its loads run on into its
// next tile and the next layer's (a cursor of its own) while the last step is consumed.  Tokens are staged once per distinct
// activation.  With few tiles K is cut over `split` warps whose sums are added in order (no longer one ascending chain).
// Bound by the warps' latencies and issue slots: 16 tokens, 0.7 GB of weights, 206 -> 190 us (3.5 TB/s) against a ring refilled
// at every tile, 32-bit fragment loads and tokens staged per layer, one load at a time.
struct MmaStreamCfg {
    static constexpr int MAX_WARPS = 16, MAX_STAGES = 4;
    static constexpr int STAGE_BYTES = 4096 + 256;
    template <int NT> static constexpr size_t smem_bytes(int max_groups, int warps, int stages, int split)
    {
        return 1024 + (size_t)warps * stages * STAGE_BYTES + MmaStep<NT, true, 32>::token_bytes(max_groups) +
               (split > 1 ? (size_t)warps * NT * 4 * 32 * 4 : 0) + MAX_WARPS * MAX_STAGES * 8 + 16;
    }
};

template <int NT, typename Params>
__global__ void __launch_bounds__(MmaStreamCfg::MAX_WARPS * 32, 1)
gemv_mma_kernel(const __grid_constant__ Params p, int stages, int early)
{
    using Cfg = MmaStreamCfg;
    using G = MmaStep<NT, true, 32>;
    extern __shared__ __align__(16) uint8_t smem[];
    const int WARPS = blockDim.x >> 5;
    uint8_t *sMant = smem + ((1024u - (ptx::smem_u32(smem) & 1023u)) & 1023u);       // [WARPS][stages][4096]
    uint8_t *sExp = sMant + WARPS * stages * G::MANT_BYTES;                            // [WARPS][stages][256]
    uint2 *sB = reinterpret_cast<uint2 *>(sExp + WARPS * stages * G::EXP_BYTES);
    const int max_groups = p.max_nb / G::GB;
    f32x2_t *sCS = reinterpret_cast<f32x2_t *>(sB + (size_t)max_groups * G::B_GROUP);
    uint8_t *sBar = reinterpret_cast<uint8_t *>(sCS + (size_t)max_groups * G::S_GROUP);   // [MAX_WARPS][MAX_STAGES] mbarriers
    volatile uint32_t *abort_flag = reinterpret_cast<volatile uint32_t *>(sBar + Cfg::MAX_WARPS * Cfg::MAX_STAGES * 8);
    float *sRed = reinterpret_cast<float *>(sBar + Cfg::MAX_WARPS * Cfg::MAX_STAGES * 8 + 16);   // [WARPS][NT * 4][32], split > 1
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    if (threadIdx.x == 0) {
        // one arrival for the TMA bytes, one per lane for its exponent bytes
        for (int i = 0; i < Cfg::MAX_WARPS * Cfg::MAX_STAGES; ++i) ptx::mbar_init(ptx::smem_u32(sBar) + 8 * i, 33);
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
    const int lo = (int)((int64_t)p.total_tiles * blockIdx.x / gridDim.x), hi = (int)((int64_t)p.total_tiles * (blockIdx.x + 1) / gridDim.x);
    int first = 0;
    while (first + 1 < p.n_layers && layers[first + 1].tile_begin <= lo) ++first;

    // end of the run of tiles from layer l on that share their staged tokens (cut at hi)
    auto segment_end = [&](int l) {
        while (l + 1 < p.n_layers && layers[l + 1].tile_begin < hi && layers[l + 1].a_mant == layers[l].a_mant &&
               layers[l + 1].w_bits == layers[l].w_bits) ++l;
        return min(hi, layers[l].tile_begin + layers[l].n_tiles);
    };
    // the load cursor: layer, tile, end of its segment; this warp's groups of the tile; the next step.  What a step needs of the
    // layer is looked up once per tile (read from the table at every step it was 17 of 42 loads and a third of the instructions)
    const uint32_t my_bar = ptx::smem_u32(sBar) + 8 * warp * Cfg::MAX_STAGES;
    const uint32_t my_mant = ptx::smem_u32(sMant) + warp * stages * G::MANT_BYTES;
    uint8_t *my_exp = sExp + warp * stages * G::EXP_BYTES;
    int c_li = first, c_seg = lo < hi ? segment_end(first) : hi, c_tile = lo + slot, c_group = 0, c_end = 0, c_stage = 0;
    int c_r0 = 0, c_nb = 0;
    const uint8_t *c_exp[2] = {nullptr, nullptr};      // exponent bytes of this lane's two rows, at its word of a group of four
    const CUtensorMap *c_map = tmaps;
    bool c_live = lo < hi;
    auto cursor_tile = [&]() {                // c_tile may be past its segment: to the first tile of this warp that has steps
        while (c_live) {
            while (c_live && c_tile >= c_seg) {
                if (c_seg >= hi) { c_live = false; break; }
                while (layers[c_li].tile_begin + layers[c_li].n_tiles <= c_seg) ++c_li;
                c_tile = c_seg + slot;
                c_seg = segment_end(c_li);
            }
            if (!c_live) return;
            while (layers[c_li].tile_begin + layers[c_li].n_tiles <= c_tile) ++c_li;
            const StreamLayer &L = layers[c_li];
            const int ng = L.K / G::KGROUP;
            c_group = ng * piece / S;
            c_end = ng * (piece + 1) / S;
            if (c_group < c_end) {
                c_r0 = (c_tile - L.tile_begin) * 16;
                c_nb = L.K >> 5;
                c_map = tmaps + 2 * c_li;
#pragma unroll
                for (int i = 0; i < 2; ++i)
                    c_exp[i] = L.w_exp + (int64_t)(min(c_r0 + (lane >> 2) + 8 * i, L.N - 1) >> L.w_rows2) * c_nb;
                return;
            }
            c_tile += TPR;
        }
    };
    auto issue = [&]() {                      // the cursor's step into stage c_stage (warp-collective), then one step on
        if (!c_live || *abort_flag != 0) return;
        const uint32_t bar = my_bar + 8 * c_stage;
        if (lane == 0) {
            const uint32_t dst = my_mant + c_stage * G::MANT_BYTES;
            ptx::mbar_arrive_expect_tx(bar, G::MANT_BYTES);
            ptx::tma_load_2d(dst, c_map, c_group * 64, c_r0, bar);               // rows >= N, bytes >= K / 2: zeros
            ptx::tma_load_2d(dst + 2048, c_map, c_group * 64 + 128, c_r0, bar);
        }
        const uint32_t dx = ptx::smem_u32(my_exp + c_stage * G::EXP_BYTES) + lane * 4;
        const int b = c_group * G::GB + (lane & 3) * 4;                          // 16 rows x 4 words; whole words (K % 128 == 0)
        const int at = b < c_nb ? b : 0, valid = b < c_nb ? 4 : 0;
        cp_async4(dx, c_exp[0] + at, valid);
        cp_async4(dx + 128, c_exp[1] + at, valid);
        cp_async_arrive(bar);
        if (++c_stage == stages) c_stage = 0;
        c_group += G::GROUPS;
        if (c_group >= c_end) {
            c_tile += TPR;
            cursor_tile();
        }
    };
    cursor_tile();
    for (int i = 0; i < stages; ++i) issue();
    if (early) ptx::dep_wait();               // the quantized tokens
    if (threadIdx.x == 0) ptx::dep_trigger();

    int st = 0;                               // stage and parity of the next step to consume
    uint32_t parity = 0;
    bool timed_out = false;
    int seg_li = first;
    for (int seg_lo = lo; seg_lo < hi;) {
        while (layers[seg_li].tile_begin + layers[seg_li].n_tiles <= seg_lo) ++seg_li;
        const int seg_hi = segment_end(seg_li);
        {
            const StreamLayer &L = layers[seg_li];
            const int nb = L.K >> 5, T = L.T;
            __syncthreads();                  // the previous segment's tokens are consumed
            // eight words of a thread in flight at once, then its scales, four at a time
            const bool nib_a = L.a_bits <= 4;
            const int words = nb * G::TP * 4, scales = nb * G::TP;
            for (int i0 = threadIdx.x; i0 < words; i0 += 8 * blockDim.x) {
                uint2 raw[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int i = i0 + u * blockDim.x, tq = i & 3, tok = (i >> 2) % G::TP, b = (i >> 2) / G::TP;
                    raw[u] = make_uint2(0u, 0u);
                    if (i < words && tok < T) {     // 8 mantissas, k = 32b + 8tq ..
                        if (nib_a) raw[u].x = __ldg(reinterpret_cast<const uint32_t *>(L.a_mant + (int64_t)tok * (L.K >> 1) + b * 16 + tq * 4));
                        else raw[u] = __ldg(reinterpret_cast<const uint2 *>(L.a_mant + (int64_t)tok * L.K + b * 32 + tq * 8));
                    }
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int i = i0 + u * blockDim.x;
                    if (i >= words) break;
                    uint32_t wlo = raw[u].x, whi = raw[u].y;
                    if (nib_a) {
                        uint32_t by[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) by[j] = (uint32_t)((((int)(raw[u].x << (28 - 4 * j))) >> 28) & 0xFF);
                        wlo = by[0] | (by[1] << 8) | (by[2] << 16) | (by[3] << 24);
                        whi = by[4] | (by[5] << 8) | (by[6] << 16) | (by[7] << 24);
                    }
                    put_token_words<NT, true>(sB, (i >> 2) / G::TP, (i >> 2) % G::TP, i & 3, wlo, whi);
                }
            }
            // 2^(Ea-127-(wa-2)) * 2^-(ww-2) * 2^-4, every factor an exact power of two
            const float unit = small_neg_pow2(L.w_bits) * 0.0625f;
            for (int i0 = threadIdx.x; i0 < scales; i0 += 4 * blockDim.x) {
                int eb[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int i = i0 + u * blockDim.x, b = i % nb, tok = i / nb;
                    eb[u] = i < scales && tok < T ? (int)__ldg(L.a_exp + (int64_t)(tok >> L.a_rows2) * nb + b) : 0;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int i = i0 + u * blockDim.x;
                    if (i < scales) reinterpret_cast<float *>(sCS)[token_scale_at<NT>(i % nb, i / nb)] = f32_scale(eb[u], L.a_bits) * unit;
                }
            }
            __syncthreads();
        }
        int li = seg_li;
        for (int base = seg_lo; base < seg_hi; base += TPR) {
            const int tile = base + slot;
            const bool active = tile < seg_hi;
            f32x2_t accA[NT], accB[NT];        // rows g / g + 8, tokens (2t, 2t + 1) of each column tile
#pragma unroll
            for (int n = 0; n < NT; ++n) accA[n] = accB[n] = pack2(0.f, 0.f);
            if (active) {
                while (layers[li].tile_begin + layers[li].n_tiles <= tile) ++li;
                const int ng = layers[li].K / G::KGROUP;
                const int g_end = ng * (piece + 1) / S;
                for (int gr = ng * piece / S; gr < g_end && !timed_out; gr += G::GROUPS) {
                    const bool ok = ptx::mbar_wait_bounded(my_bar + 8 * st, parity, abort_flag, STREAM_WAIT_LIMIT_NS);
                    if (!__all_sync(0xFFFFFFFFu, ok)) {
                        timed_out = true;
                        *abort_flag = 1;      // the other warps stop issuing as well
                        break;
                    }
                    mma_step<NT, true, 32>(my_mant + st * G::MANT_BYTES, my_exp + st * G::EXP_BYTES, sB + (size_t)gr * G::B_GROUP,
                                           sCS + (size_t)gr * G::S_GROUP, min(g_end - gr, G::GROUPS), lane, accA, accB);
                    __syncwarp();             // every lane is done reading the stage
                    if (++st == stages) { st = 0; parity ^= 1u; }
                    if (lane == 0) ptx::fence_proxy_async_smem();
                    issue();
                }
            }
            float acc[NT][4];
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                unpack2(accA[n], acc[n][0], acc[n][1]);
                unpack2(accB[n], acc[n][2], acc[n][3]);
            }
            if (S > 1) {                      // CTA-uniform
                __syncthreads();
#pragma unroll
                for (int n = 0; n < NT; ++n)
#pragma unroll
                    for (int j = 0; j < 4; ++j) sRed[((warp * NT + n) * 4 + j) * 32 + lane] = acc[n][j];
                __syncthreads();
                if (piece == 0 && active) {
#pragma unroll
                    for (int n = 0; n < NT; ++n)
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            for (int q = 1; q < S; ++q) acc[n][j] += sRed[(((warp + q) * NT + n) * 4 + j) * 32 + lane];
                }
            }
            if (active && piece == 0) {
                const StreamLayer &L = layers[li];
                const int r0 = (tile - L.tile_begin) * 16;
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
        // (a warp whose wait expired goes through the remaining rounds without steps: the CTA's barriers stay matched)
        seg_lo = seg_hi;
    }
    if (timed_out) atomicOr(p.status, 1u);
    if (*abort_flag != 0) {                   // copies already in flight get time to land before the shared memory is released
        const uint64_t t0 = ptx::globaltimer_ns();
        while (ptx::globaltimer_ns() - t0 < 100000ull) __nanosleep(1000);
    }
    __syncthreads();
}

// ---- one layer, one launch ---------------------------------------------------------------------------
// A cluster of C CTAs owns row groups of 8 warps x 16 rows; each CTA takes a C-th of K.  So a CTA quantizes only its own slice
// of the tokens (into the operand form, in shared memory: no launch in front, nothing in global memory) while its first weight
// stages are on their way, and the partial sums are added in slice order through distributed shared memory at the end.
// Takes blocks of 16 and 32, weights of 2 to 8 bits in container form with rows of whole 16 bytes, two-row weight blocks.
struct GemvArgs {
    const void *x;
    int64_t ldx;
    const uint8_t *w_exp;
    const float *bias;            // nullable
    float *y;                     // [T, ldy]
    int64_t ldy;
    int T, N, K;
    int a_bits, w_bits, w_rows2;
    int rounds;                   // row groups per cluster
    int row_groups;               // ceil(N / 128)
    int bf16;                     // type of x
    int exp_words;                // 1: every step's exponent bytes are whole aligned words
    int max_groups;               // largest slice of K, in groups
    uint32_t *status;
};

struct GemvCfg {
    static constexpr int WARPS = 8, THREADS = WARPS * 32, MAX_STAGES = 4, MAX_CLUSTER = 8;
    static constexpr int ROWS = WARPS * 16;
    static constexpr int PITCH = ROWS + 4;                       // floats between tokens of a partial tile: conflict-free
    template <int NT, bool NIB, int BLOCK> static constexpr size_t smem_bytes(int max_groups, int stages, int rounds, int cluster)
    {
        using G = MmaStep<NT, NIB, BLOCK>;
        const size_t staged = (size_t)WARPS * stages * (G::MANT_BYTES + G::EXP_BYTES) + G::token_bytes(max_groups);
        const size_t part = cluster > 1 ? (size_t)rounds * G::TP * PITCH * 4 : 0;
        // one round: the partial tile takes the place of the consumed stages and tokens
        return 2048 + (rounds == 1 ? (staged > part ? staged : part) : staged + part);
    }
};

__device__ __forceinline__ float ld_shared_cluster(uint32_t addr)
{
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}

// Eight values of x from element `at` on.
__device__ __forceinline__ void load_x8(const GemvArgs &p, int64_t at, float (&v)[8])
{
    if (p.bf16) Load8<__nv_bfloat16>::run(static_cast<const __nv_bfloat16 *>(p.x) + at, v);
    else Load8<float>::run(static_cast<const float *>(p.x) + at, v);
}

template <int NT, bool NIB, int BLOCK>
__global__ void __launch_bounds__(GemvCfg::THREADS, 2)
gemv_single_kernel(const __grid_constant__ CUtensorMap tm, const GemvArgs p, int stages)
{
    using Cfg = GemvCfg;
    using G = MmaStep<NT, NIB, BLOCK>;
    constexpr int WARPS = Cfg::WARPS, PITCH = Cfg::PITCH;
    extern __shared__ __align__(16) uint8_t smem[];
    uint8_t *sBase = smem + ((1024u - (ptx::smem_u32(smem) & 1023u)) & 1023u);
    uint8_t *sBar = sBase;                                                            // barriers, then 1024-byte aligned stages
    volatile uint32_t *abort_flag = reinterpret_cast<volatile uint32_t *>(sBar + WARPS * Cfg::MAX_STAGES * 8);
    uint8_t *sMant = sBase + 1024;
    uint8_t *sExp = sMant + WARPS * stages * G::MANT_BYTES;
    uint2 *sB = reinterpret_cast<uint2 *>(sExp + WARPS * stages * G::EXP_BYTES);
    f32x2_t *sCS = reinterpret_cast<f32x2_t *>(sB + (size_t)p.max_groups * G::B_GROUP);
    // [rounds][TP][PITCH]
    float *sPart = reinterpret_cast<float *>(p.rounds == 1 ? sMant : reinterpret_cast<uint8_t *>(sCS + (size_t)p.max_groups * G::S_GROUP));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int rank = (int)ptx::cluster_ctarank(), C = (int)ptx::cluster_nctarank();
    if (threadIdx.x == 0) {
        for (int i = 0; i < WARPS * Cfg::MAX_STAGES; ++i) ptx::mbar_init(ptx::smem_u32(sBar) + 8 * i, 33);
        *abort_flag = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tm);
    }
    __syncthreads();
    ptx::dep_wait();
    if (threadIdx.x == 0) ptx::dep_trigger();

    const int row_bytes = NIB ? p.K >> 1 : p.K, nb = p.K / BLOCK;
    const int ng = (row_bytes + 63) >> 6;
    const int g_lo = ng * rank / C, g_hi = ng * (rank + 1) / C;                 // this CTA's groups
    const int first = (int)(blockIdx.x / C) * p.rounds;                           // its cluster's first row group
    const int rounds = min(p.rounds, p.row_groups - first);
    const uint32_t my_bar = ptx::smem_u32(sBar) + 8 * warp * Cfg::MAX_STAGES;
    const uint32_t my_mant = ptx::smem_u32(sMant) + warp * stages * G::MANT_BYTES;
    uint8_t *my_exp = sExp + warp * stages * G::EXP_BYTES;

    int c_round = 0, c_group = g_lo, c_stage = 0;
    auto issue = [&]() {                      // the load cursor's step (round, group) into stage c_stage, then one step on
        const int r0 = (first + c_round) * Cfg::ROWS + warp * 16;
        if (c_round >= rounds || r0 >= p.N || c_group >= g_hi || *abort_flag != 0) return;
        const uint32_t bar = my_bar + 8 * c_stage;
        if (lane == 0) {
            const uint32_t dst = my_mant + c_stage * G::MANT_BYTES;
            ptx::mbar_arrive_expect_tx(bar, G::MANT_BYTES);
            ptx::tma_load_2d(dst, &tm, c_group * 64, r0, bar);                   // rows >= N, bytes past the row's end: zeros
            ptx::tma_load_2d(dst + 2048, &tm, c_group * 64 + 128, r0, bar);
        }
        uint8_t *dx = my_exp + c_stage * G::EXP_BYTES;                           // [16 rows][4 * GB]
        const int b0 = c_group * G::GB;
#pragma unroll
        for (int i = 0; i < G::EXP_BYTES / 128; ++i) {
            const int w = lane + 32 * i, r = w / G::GB, b = b0 + (w % G::GB) * 4;
            const uint8_t *src = p.w_exp + (int64_t)(min(r0 + r, p.N - 1) >> p.w_rows2) * nb;
            if (p.exp_words) {
                cp_async4(ptx::smem_u32(dx) + w * 4, b < nb ? src + b : src, b < nb ? 4 : 0);
            } else {
                uint32_t v = 0;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (b + j < nb) v |= (uint32_t)__ldg(src + b + j) << (8 * j);
                reinterpret_cast<uint32_t *>(dx)[w] = v;
            }
        }
        if (p.exp_words) cp_async_arrive(bar);
        else ptx::mbar_arrive(bar);
        if (++c_stage == stages) c_stage = 0;
        c_group += G::GROUPS;
        if (c_group >= g_hi) {
            c_group = g_lo;
            ++c_round;
        }
    };
    for (int i = 0; i < stages; ++i) issue();

    // this CTA's slice of the tokens: a warp takes (token, 256 k) items, a lane 8 k; the quantizer's rounding
    {
        const int k_lo = g_lo * G::KGROUP, k_pad = (g_hi - g_lo) * G::KGROUP;
        const int segs = (k_pad + 255) >> 8;
        const float unit = small_neg_pow2(p.w_bits) * (NIB ? 0.0625f : 1.f);     // the weights' binary point, the nibbles' 16
        // four items of a warp in flight at once: one after the other they are a chain of memory latencies (16 tokens of
        // 11008 x 4096 21.4 -> 19.4 us, 32 of 4096 x 4096 16.0 -> 13.8)
        constexpr int U = 4;
        for (int i0 = warp; i0 < G::TP * segs; i0 += U * WARPS) {
            float v[U][8];
            int tok[U], ks[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = i0 + u * WARPS;
                tok[u] = i / segs;
                ks[u] = (i - tok[u] * segs) * 256 + 8 * lane;
                if (tok[u] < p.T && k_lo + ks[u] < p.K && ks[u] < k_pad) {
                    load_x8(p, (int64_t)tok[u] * p.ldx + k_lo + ks[u], v[u]);
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[u][j] = 0.f;
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                uint2 q = make_uint2(0u, 0u);
                float scale = 0.f;
                if (tok[u] < p.T) {           // warp-uniform
                    float am = 0.f;
#pragma unroll
                    for (int j = 0; j < 8; ++j) am = absmax_nan(am, v[u][j]);
                    uint32_t amax = __float_as_uint(am);
#pragma unroll
                    for (int d = 1; d < BLOCK / 8; d <<= 1) amax = max(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, d));
                    const int ebyte = (int)(amax >> 23);
                    q = encode8_bytes(v[u], ebyte, p.a_bits);
                    scale = f32_scale(ebyte, p.a_bits) * unit;
                }
                if (tok[u] < G::TP && ks[u] < k_pad) {
                    put_token_words<NT, NIB>(sB, ks[u] >> 5, tok[u], lane & 3, q.x, q.y);
                    if ((lane & (BLOCK / 8 - 1)) == 0)
                        reinterpret_cast<float *>(sCS)[token_scale_at<NT>(ks[u] / BLOCK, tok[u])] = scale;
                }
            }
        }
    }
    __syncthreads();

    int st = 0;
    uint32_t parity = 0;
    bool timed_out = false;
    for (int r = 0; r < rounds; ++r) {
        const int r0 = (first + r) * Cfg::ROWS + warp * 16;
        f32x2_t accA[NT], accB[NT];
#pragma unroll
        for (int n = 0; n < NT; ++n) accA[n] = accB[n] = pack2(0.f, 0.f);
        for (int gr = g_lo; gr < g_hi && r0 < p.N && !timed_out; gr += G::GROUPS) {
            const bool ok = ptx::mbar_wait_bounded(my_bar + 8 * st, parity, abort_flag, STREAM_WAIT_LIMIT_NS);
            if (!__all_sync(0xFFFFFFFFu, ok)) {
                timed_out = true;
                *abort_flag = 1;
                break;
            }
            mma_step<NT, NIB, BLOCK>(my_mant + st * G::MANT_BYTES, my_exp + st * G::EXP_BYTES, sB + (size_t)(gr - g_lo) * G::B_GROUP,
                                     sCS + (size_t)(gr - g_lo) * G::S_GROUP, min(g_hi - gr, G::GROUPS), lane, accA, accB);
            __syncwarp();                     // every lane is done reading the stage
            if (++st == stages) { st = 0; parity ^= 1u; }
            if (lane == 0) ptx::fence_proxy_async_smem();
            issue();
        }
        float acc[NT][4];
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            unpack2(accA[n], acc[n][0], acc[n][1]);
            unpack2(accB[n], acc[n][2], acc[n][3]);
        }
        if (C > 1 && p.rounds == 1) __syncthreads();     // the partial tile overwrites the stages and tokens
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int row = g + (j >> 1) * 8, tok = n * 8 + 2 * t + (j & 1);
                if (C > 1) sPart[(r * G::TP + tok) * PITCH + warp * 16 + row] = acc[n][j];
                else if (r0 + row < p.N && tok < p.T)
                    p.y[(int64_t)tok * p.ldy + r0 + row] = p.bias ? acc[n][j] + __ldg(p.bias + r0 + row) : acc[n][j];
            }
    }
    if (timed_out) atomicOr(p.status, 1u);
    if (*abort_flag != 0) {                   // copies already in flight get time to land before the shared memory is released
        const uint64_t t0 = ptx::globaltimer_ns();
        while (ptx::globaltimer_ns() - t0 < 100000ull) __nanosleep(1000);
    }
    __syncthreads();
    if (C > 1) {
        // (round, token) items dealt to the CTAs; a thread adds one row's C partial sums in slice order
        ptx::cluster_sync();
        const uint32_t part = ptx::smem_u32(sPart);
        const int row = threadIdx.x % Cfg::ROWS, half = threadIdx.x / Cfg::ROWS;
        for (int i = rank + C * half; i < rounds * p.T; i += 2 * C) {
            const int r = i / p.T, tok = i - r * p.T, n = (first + r) * Cfg::ROWS + row;
            const uint32_t at = part + (uint32_t)(((r * G::TP + tok) * PITCH + row) * 4);
            float v[Cfg::MAX_CLUSTER];
#pragma unroll
            for (int c = 0; c < Cfg::MAX_CLUSTER; ++c)
                if (c < C) v[c] = ld_shared_cluster(ptx::map_to_cta(at, c));
            float sum = v[0];
#pragma unroll
            for (int c = 1; c < Cfg::MAX_CLUSTER; ++c)
                if (c < C) sum += v[c];
            if (n < p.N) p.y[(int64_t)tok * p.ldy + n] = p.bias ? sum + __ldg(p.bias + n) : sum;
        }
        ptx::cluster_sync();                  // nobody leaves while its shared memory is read
    }
}

}  // namespace mx
