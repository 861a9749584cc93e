// Operands of the block-scaled product in records: the layout that the tensor pipe's block-scaled
// 8-bit MMA (kind::mxf8f6f4, one E8M0 scale per 32 elements along K) reads without any rearrangement.
//
// An operand [rows, K] is cut into records of 128 rows x 128 k.  Record (panel, kb) is 16 KB of E4M3 bytes in the
// canonical K-major shape without swizzle -- [8 chunks of 16 k][128 rows][16 bytes], so a chunk of 8 rows is
// 128 contiguous bytes and a record one contiguous copy -- and records follow one another along K.
//
// Scales.  A row has ONE scale per record: byte S, 2^(S-127), and its elements are q * 2^t with
// t = E - (w-2) - (S-127) per block.  E4M3 holds q * 2^t without rounding for |q| <= 16 (mantissa widths up to 5) as long as
// t >= -9 and |q| * 2^t <= 448; S is set by the largest exponent of the row's blocks in the record, with t at its upper
// limit there (5 for nibble containers, |q| <= 8, else 4), so the blocks of a record may lie up to 14 (13) binades apart.  One scale per 128 k instead of
// the hardware's one per 32 means that the four bytes of a tensor-memory cell serve four K steps: the copies
// shared -> tensor memory, which the tensor pipe executes between MMAs (about 60 ns per K step of 0.35 us when done for
// each one), are needed for every fourth step only.  They lie in chunks of 512 bytes, byte
// (row % 32) * 16 + (row / 32) * 4 + kb % 4 -- what tcgen05.cp.32x128b.warpx4 puts where the MMA looks -- in the order
// [kb / 4][panel], so that a tile's two panels of W are adjacent.
//
// Where the blocks of some row and record lie further apart, each of them keeps a scale of its own and the flag byte of
// the record's 8 rows is set: the product then takes the halves (16 k) of every 32 k of this K step in separate MMAs with
// their own scales, which are written for every row into a second array: 1 KB per record, order
// [kb][panel], one chunk for the k % 32 < 16 and one for the others, byte
// (row % 32) * 16 + (row / 32) * 4 + (k / 32) % 4.  Every flag byte has one writer, so nothing is cleared between calls.
//
// The passes are bound by HBM and, at a few thousand rows, by the latency of their few iterations.  A quantizing
// lane owns 16 consecutive k of a row (so a block of 16 needs no exchange and one of 32 a single shuffle) and eight
// lanes with neighbouring rows store 128 contiguous bytes; four 16-byte loads per lane and half record are in flight
// at once.  A decoding lane owns 32 consecutive k.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "mx_ptx.cuh"
#include "mx_quantize.cuh"

namespace mx {

constexpr int REC_ROWS = 128, REC_K = 128;
constexpr uint32_t REC_BYTES = REC_ROWS * REC_K;         // E4M3 bytes of a record
constexpr uint32_t REC_SF_BYTES = 512;                   // scales of 128 rows x 4 records
constexpr uint32_t REC_SFW_BYTES = 1024;                 // scales of one record's half blocks

struct RecOut {
    uint8_t *elems;          // [panels][kblocks][REC_BYTES]
    uint8_t *sf;             // [ceil(kblocks / 4)][panels_sf][REC_SF_BYTES]
    uint8_t *sf_wide;        // [kblocks][panels_sf][REC_SFW_BYTES]
    uint8_t *flags;          // [panels][kblocks][16], one byte per 8 rows: 1 = some row's blocks keep scales of their own
    int panels, panels_sf, kblocks;
};

// Largest t with |element| * 2^t <= 256 < 448 (the E4M3 maximum) for every q the container holds (-8 and -16 included).
__device__ __forceinline__ int rec_t_max(int w) { return w <= 4 ? 5 : 4; }
constexpr int REC_T_MIN = -9;                            // multiples of 2^-9 are E4M3 numbers (up to 4 significant bits)

// Scale byte of a block with exponent byte e (finite): 2^(S-127) with the block's elements q * 2^t, t <= t_max.
__device__ __forceinline__ int rec_scale_byte(int e, int w) { return max(0, e - (w - 2) - rec_t_max(w)); }

// The scale of a row in one record, agreed on by the LANES neighbouring lanes that hold the row.  e0, e1: exponent bytes
// of the lane's two groups of 16 k; z0, z1: the group holds zeros only (its exponent does not matter).
struct RecScale { int s, s0, s1; bool wide; };           // the row's byte; the bytes the two groups are scaled by

template <int LANES = 4>
__device__ __forceinline__ RecScale rec_scales(int e0, int e1, bool z0, bool z1, int w)
{
    // largest exponent in the low half word, 255 - smallest in the high one: one shuffle and one maximum per step
    uint32_t m = (z0 ? 0u : (uint32_t)e0 | ((uint32_t)(255 - e0) << 16));
    m = __vmaxu2(m, z1 ? 0u : (uint32_t)e1 | ((uint32_t)(255 - e1) << 16));
#pragma unroll
    for (int d = 1; d < LANES; d <<= 1) m = __vmaxu2(m, __shfl_xor_sync(0xFFFFFFFFu, m, d));
    const int hi = (int)(m & 0xFFFFu), lo = 255 - (int)(m >> 16);
    RecScale r;
    r.wide = false;
    r.s = hi == 255 ? 255 : rec_scale_byte(hi, w);       // Inf/NaN: the row's results are NaN whatever the rest holds
    r.s0 = r.s1 = r.s;
    if (hi != 255 && lo - (w - 2) - r.s < REC_T_MIN) {
        r.wide = true;
        r.s0 = rec_scale_byte(z0 ? 0 : e0, w);
        r.s1 = rec_scale_byte(z1 ? 0 : e1, w);
    }
    return r;
}

// 2^(127 - S); S <= 254 - t_max
__device__ __forceinline__ float rec_inv_scale(int s) { return __uint_as_float((uint32_t)(254 - s) << 23); }

__device__ __forceinline__ uint32_t e4m3x2(float lo, float hi)
{
    uint16_t r;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ uint32_t e4m3x4(float a, float b, float c, float d) { return e4m3x2(a, b) | (e4m3x2(c, d) << 16); }

// The scale byte of the row and record.
__device__ __forceinline__ void rec_store_scale(const RecOut &o, int panel, int kb, int rp, int s)
{
    o.sf[((int64_t)(kb >> 2) * o.panels_sf + panel) * REC_SF_BYTES + (rp & 31) * 16 + (rp >> 5) * 4 + (kb & 3)] = (uint8_t)s;
}
// The scale bytes of its groups g0 and g1 of 16 k (numbers within the record).  Where none of the warp's rows is wide all
// eight bytes of a row are its one scale: two lanes write them as words (c4 = number of the lane among its row's four).
__device__ __forceinline__ void rec_store_wide(const RecOut &o, int panel, int kb, int rp, const RecScale &s, bool wide, int c4, int g0, int g1)
{
    uint8_t *d = o.sf_wide + ((int64_t)kb * o.panels_sf + panel) * REC_SFW_BYTES + (rp & 31) * 16 + (rp >> 5) * 4;
    if (!wide) {
        if (c4 < 2) *reinterpret_cast<uint32_t *>(d + 512 * c4) = (uint32_t)s.s * 0x01010101u;
        return;
    }
    d[(g0 & 1) * 512 + (g0 >> 1)] = (uint8_t)s.s0;
    d[(g1 & 1) * 512 + (g1 >> 1)] = (uint8_t)s.s1;
}

// Eight values of one block (exponent byte e, width w) -> E4M3 codes of q * 2^t, t = e - (w-2) - sb.  The sum x + M
// rounds x to a multiple of the block's step exactly as in encode8_full; one fma takes M off again and applies the
// power of two (both exact), one instruction clamps the magnitude to qmax * 2^t.  Blocks near the top of the range
// (M not finite) take encode8_full.
__device__ __forceinline__ uint2 rec_encode8(const float (&v)[8], int e, int w, int sb)
{
    float q[8];
    if (e <= 229 + w) {
        const int t = e - (w - 2) - sb;
        const float M = __uint_as_float(((uint32_t)(e + 25 - w) << 23) | 0x00400000u);
        const float inv = rec_inv_scale(sb);
        const float mi = __uint_as_float(((uint32_t)(t + 150) << 23) | 0x00400000u);        // M * inv = 1.5 * 2^(23+t)
        const float lim = (float)((1 << (w - 1)) - 1) * __uint_as_float((uint32_t)(t + 127) << 23);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float r = fmaf(v[i] + M, inv, -mi);
            asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(q[i]) : "f"(r), "f"(lim));
        }
    } else {
        const float inv = rec_inv_scale(min(sb, 254));
        float xh[8];
        encode8_full(v, e, w, xh);
#pragma unroll
        for (int i = 0; i < 8; ++i) q[i] = xh[i] * inv;
    }
    return make_uint2(e4m3x4(q[0], q[1], q[2], q[3]), e4m3x4(q[4], q[5], q[6], q[7]));
}

constexpr uint32_t E4M3_NAN4 = 0x7F7F7F7Fu;

// Sixteen values of one block -> their 16 bytes.
__device__ __forceinline__ uint4 rec_encode16(const float (&v)[2][8], int e, bool zero, int w, int sb)
{
    if (sb == 255) return make_uint4(E4M3_NAN4, E4M3_NAN4, E4M3_NAN4, E4M3_NAN4);
    if (zero) return make_uint4(0, 0, 0, 0);
    const uint2 x = rec_encode8(v[0], e, w, sb), y = rec_encode8(v[1], e, w, sb);
    return make_uint4(x.x, x.y, y.x, y.y);
}

// Floating-point rows -> records.  Warp item = 8 rows x one record's 128 k; lane = row * 4 + chunk, two passes of four
// chunks.  ROWS2: rows 2i and 2i + 1 share the exponents.  Rows >= `rows` and k >= K become
// zeros.
template <typename InT, int BLOCK, bool ROWS2>
__device__ __forceinline__ void rec_quantize_body(const InT *__restrict__ x, int64_t rows, int64_t K, int64_t ldx, int w,
                                                  const RecOut &o, uint32_t warp_id, uint32_t n_warps)
{
    const int lane = threadIdx.x & 31, r8 = lane >> 2, c4 = lane & 3;
    const uint32_t kblocks = (uint32_t)o.kblocks, items = (uint32_t)o.panels * (REC_ROWS / 8) * kblocks;
    for (uint32_t it = warp_id; it < items; it += n_warps) {
        // neighbouring warps take neighbouring records of the same rows
        const uint32_t grp = it / kblocks;
        const int kb = (int)(it - grp * kblocks);
        const int64_t row = (int64_t)grp * 8 + r8;
        const int panel = (int)(grp >> 4), rp = (int)(row & 127);
        float v[2][2][8];
        const InT *src = x + row * ldx + kb * REC_K + c4 * 16;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (row < rows && (int64_t)kb * REC_K + u * 64 + c4 * 16 < K) {
                Load8<InT>::run(src + u * 64, v[u][0]);
                Load8<InT>::run(src + u * 64 + 8, v[u][1]);
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) v[u][0][i] = v[u][1][i] = 0.f;
            }
        }
        int e[2];
        bool z[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            float am = 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i) am = absmax_nan(absmax_nan(am, v[u][0][i]), v[u][1][i]);
            uint32_t amax = __float_as_uint(am);
            if (ROWS2) amax = max(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, 4));
            if (BLOCK == 32) amax = max(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, 1));
            e[u] = (int)(amax >> 23);
            z[u] = amax == 0;
        }
        const RecScale s = rec_scales(e[0], e[1], z[0], z[1], w);
        uint8_t *dst = o.elems + ((int64_t)panel * kblocks + kb) * REC_BYTES + c4 * (REC_ROWS * 16) + rp * 16;
#pragma unroll
        for (int u = 0; u < 2; ++u)
            *reinterpret_cast<uint4 *>(dst + u * 4 * (REC_ROWS * 16)) = rec_encode16(v[u], e[u], z[u], w, u ? s.s1 : s.s0);
        if (c4 == 0) rec_store_scale(o, panel, kb, rp, s.s);
        const bool wide = __any_sync(0xFFFFFFFFu, s.wide);
        rec_store_wide(o, panel, kb, rp, s, wide, c4, c4, 4 + c4);
        if (lane == 0) o.flags[((int64_t)panel * kblocks + kb) * 16 + (grp & 15)] = wide;
    }
}

// Four table lookups at once: nibble i of `sel` (two's complement) picks byte i of the result, from p0 p1 for 0..7 and from
// n0 n1 for -8..-1 (a byte permute selects by three bits).  The p entries have sign bit 0, the n entries 1.
__device__ __forceinline__ uint32_t rec_lut4(uint32_t sel, uint32_t p0, uint32_t p1, uint32_t n0, uint32_t n1)
{
    const uint32_t pos = __byte_perm(p0, p1, sel & 0x7777u), neg = __byte_perm(n0, n1, sel & 0x7777u);
    uint32_t keep;                      // selector bit 3 copies the sign of the selected byte: 0x7F for q >= 0, 0 for q < 0
    asm("prmt.b32 %0, %1, %1, %2;" : "=r"(keep) : "r"(0x7F7F7F7Fu), "r"(sel));
    return ((pos & keep) | (neg & ~keep)) ^ ((keep << 1) & 0x80808080u);
}

// Sixteen mantissas of one block -> E4M3 codes of q * 2^t.
// Nibbles by table: the codes of t = 0 plus t in every exponent field (but that of zero), which holds while the smallest
// value is a normal E4M3 number (t >= -6).  Other t, and int8 mantissas: the offset integer as a float in
// [2^23, 2^23 + 255], one exact fma, one conversion.
template <bool NIBBLE>
__device__ __forceinline__ uint4 rec_codes16(const uint32_t (&m)[NIBBLE ? 2 : 4], int t)
{
    uint32_t b[4];
    if (NIBBLE && t >= -6) {
        const uint32_t dt = (uint32_t)t * 0x08080808u;
        const uint32_t p0 = 0x44403800u + (uint32_t)t * 0x08080800u, p1 = 0x4E4C4A48u + dt;      // 0 1 2 3, 4 5 6 7
        const uint32_t n0 = 0xCACCCED0u + dt, n1 = 0xB8C0C4C8u + dt;                             // -8 .. -5, -4 .. -1
#pragma unroll
        for (int i = 0; i < 4; ++i) b[i] = rec_lut4(i & 1 ? m[i >> 1] >> 16 : m[i >> 1], p0, p1, n0, n1);
    } else {
        const float f = __uint_as_float((uint32_t)(127 + t) << 23);
        const float c = (NIBBLE ? -8388616.0f : -8388736.0f) * f;        // -(2^23 + 8), -(2^23 + 128)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float q[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                uint32_t u;
                if (NIBBLE) u = ((((i & 1 ? m[i >> 1] >> 16 : m[i >> 1]) ^ 0x8888u) >> (4 * j)) & 0xFu) | 0x4B000000u;
                else u = __byte_perm(m[NIBBLE ? 0 : i] ^ 0x80808080u, 0x4B000000u, 0x7540 | j);
                q[j] = fmaf(__uint_as_float(u), f, c);
            }
            b[i] = e4m3x4(q[0], q[1], q[2], q[3]);
        }
    }
    return make_uint4(b[0], b[1], b[2], b[3]);
}

// Packed rows (container form) -> records.  Lane = row * 4 + block of 32 k; an item is UNROLL records of the same 8
// rows.  K % 32 == 0.  row_shift = 1: two-row blocks.
struct RecPacked {
    const uint8_t *mant, *exps;
    int64_t rows, K;
    int block, w, row_shift;
};

template <bool NIBBLE, int UNROLL> struct RecPackedItem {
    uint4 m[UNROLL][NIBBLE ? 1 : 2];
    uint32_t e[UNROLL];
};

template <bool NIBBLE, int UNROLL>
__device__ __forceinline__ void rec_fetch(const RecPacked &j, uint32_t it, uint32_t steps, uint32_t items, RecPackedItem<NIBBLE, UNROLL> &d)
{
    const int lane = threadIdx.x & 31, r8 = lane >> 2, c4 = lane & 3;
    const bool b16 = j.block == 16;
    const uint32_t grp = it / steps;
    const int kb0 = (int)(it - grp * steps) * UNROLL;
    const int64_t row = (int64_t)grp * 8 + r8;
    const int64_t k0 = (int64_t)kb0 * REC_K + c4 * 32;
    const uint8_t *src = j.mant + row * (NIBBLE ? j.K >> 1 : j.K) + (NIBBLE ? k0 >> 1 : k0);
    const uint8_t *ep = j.exps + (row >> j.row_shift) * (b16 ? j.K >> 4 : j.K >> 5) + (b16 ? k0 >> 4 : k0 >> 5);
    const bool live = it < items && row < j.rows;
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
#pragma unroll
        for (int i = 0; i < (NIBBLE ? 1 : 2); ++i) d.m[u][i] = make_uint4(0, 0, 0, 0);
        d.e[u] = 0;
        if (live && k0 + u * REC_K < j.K) {
#pragma unroll
            for (int i = 0; i < (NIBBLE ? 1 : 2); ++i)
                d.m[u][i] = __ldcs(reinterpret_cast<const uint4 *>(src + u * (NIBBLE ? REC_K / 2 : REC_K)) + i);
            const uint8_t *eu = ep + u * (b16 ? REC_K / 16 : REC_K / 32);
            d.e[u] = b16 ? (uint32_t)eu[0] | ((uint32_t)eu[1] << 8) : (uint32_t)eu[0] * 0x0101u;
        }
    }
}

template <bool NIBBLE, int UNROLL>
__device__ __forceinline__ void rec_convert(const RecPacked &j, const RecOut &o, uint32_t it, uint32_t steps,
                                            const RecPackedItem<NIBBLE, UNROLL> &d)
{
    const int lane = threadIdx.x & 31, r8 = lane >> 2, c4 = lane & 3;
    const uint32_t grp = it / steps;
    const int kb0 = (int)(it - grp * steps) * UNROLL;
    const int panel = (int)(grp >> 4), rp = (int)((grp * 8 + r8) & 127);
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
        const int kb = kb0 + u;
        if (kb >= o.kblocks) break;                                          // warp-uniform
        const int e0 = (int)(d.e[u] & 0xFF), e1 = (int)(d.e[u] >> 8);
        constexpr int H = NIBBLE ? 2 : 4;                                    // words per group of 16
        const uint32_t words[8] = {d.m[u][0].x, d.m[u][0].y, d.m[u][0].z, d.m[u][0].w, d.m[u][NIBBLE ? 0 : 1].x,
                                   d.m[u][NIBBLE ? 0 : 1].y, d.m[u][NIBBLE ? 0 : 1].z, d.m[u][NIBBLE ? 0 : 1].w};
        uint32_t half[2][H];
        uint32_t any[2] = {0u, 0u};
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < H; ++i) any[h] |= (half[h][i] = words[h * H + i]);
        // a block that held Inf/NaN is stored as byte 255 with zero mantissas: it still poisons
        const RecScale s = rec_scales(e0, e1, any[0] == 0 && e0 != 255, any[1] == 0 && e1 != 255, j.w);
        uint8_t *dst = o.elems + ((int64_t)panel * o.kblocks + kb) * REC_BYTES + (c4 * 2) * (REC_ROWS * 16) + rp * 16;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int sb = h ? s.s1 : s.s0;
            uint4 b = make_uint4(0, 0, 0, 0);
            if (sb == 255) b = make_uint4(E4M3_NAN4, E4M3_NAN4, E4M3_NAN4, E4M3_NAN4);
            else if (any[h]) b = rec_codes16<NIBBLE>(half[h], (h ? e1 : e0) - (j.w - 2) - sb);
            *reinterpret_cast<uint4 *>(dst + h * (REC_ROWS * 16)) = b;
        }
        if (c4 == 0) rec_store_scale(o, panel, kb, rp, s.s);
        const bool wide = __any_sync(0xFFFFFFFFu, s.wide);
        rec_store_wide(o, panel, kb, rp, s, wide, c4, 2 * c4, 2 * c4 + 1);
        if (lane == 0) o.flags[((int64_t)panel * o.kblocks + kb) * 16 + (grp & 15)] = wide;
    }
}

__device__ __forceinline__ uint32_t rec_steps(const RecOut &o, int unroll) { return (uint32_t)((o.kblocks + unroll - 1) / unroll); }

// The rest of a warp's items; `d` holds its first one.  The next item's loads are in flight under each conversion.
template <bool NIBBLE, int UNROLL>
__device__ __forceinline__ void rec_decode_body(const RecPacked &j, const RecOut &o, uint32_t warp_id, uint32_t n_warps,
                                                RecPackedItem<NIBBLE, UNROLL> &d)
{
    const uint32_t steps = rec_steps(o, UNROLL), items = (uint32_t)o.panels * (REC_ROWS / 8) * steps;
    for (uint32_t it = warp_id; it < items; it += n_warps) {
        RecPackedItem<NIBBLE, UNROLL> next;
        rec_fetch<NIBBLE, UNROLL>(j, it + n_warps, steps, items, next);
        rec_convert<NIBBLE, UNROLL>(j, o, it, steps, d);
        d = next;
    }
}

// Both operands of a layer in one launch: every warp takes its share of the activations, then of the weights.
struct RecPrepJob {
    const void *x;            // activations [M, K], leading dimension ldx
    int64_t M, K, ldx;
    int wa, block, a_rows2;
    RecPacked pw;             // weights
    RecOut a, w;
};

template <typename InT, bool NIBBLE>
__global__ void __launch_bounds__(256, 3)
rec_prep_kernel(const RecPrepJob j)
{
    ptx::dep_wait();
    ptx::dep_trigger();
    const uint32_t warps = blockDim.x >> 5;
    const uint32_t wid = blockIdx.x * warps + (threadIdx.x >> 5), nw = gridDim.x * warps;
    // the weights' items are dealt on from where the activations' end, so that no warp has more than one item above the mean
    const uint32_t ww = after_items(wid, nw, (uint32_t)j.a.panels * (REC_ROWS / 8) * (uint32_t)j.a.kblocks);
    // the first weights are on their way while the activations are quantized
    constexpr int UNROLL = 2;
    RecPackedItem<NIBBLE, UNROLL> d;
    const uint32_t steps = rec_steps(j.w, UNROLL);
    rec_fetch<NIBBLE, UNROLL>(j.pw, ww, steps, (uint32_t)j.w.panels * (REC_ROWS / 8) * steps, d);
    const InT *x = static_cast<const InT *>(j.x);
    if (j.block == 16) {
        if (j.a_rows2) rec_quantize_body<InT, 16, true>(x, j.M, j.K, j.ldx, j.wa, j.a, wid, nw);
        else rec_quantize_body<InT, 16, false>(x, j.M, j.K, j.ldx, j.wa, j.a, wid, nw);
    } else {
        if (j.a_rows2) rec_quantize_body<InT, 32, true>(x, j.M, j.K, j.ldx, j.wa, j.a, wid, nw);
        else rec_quantize_body<InT, 32, false>(x, j.M, j.K, j.ldx, j.wa, j.a, wid, nw);
    }
    rec_decode_body<NIBBLE, UNROLL>(j.pw, j.w, ww, nw, d);
}

// The same for two packed operands.
struct RecPairJob {
    RecPacked pa, pw;
    RecOut a, w;
};

template <bool NIB_A, bool NIB_W>
__global__ void __launch_bounds__(256, 3)
rec_pair_kernel(const RecPairJob j)
{
    ptx::dep_wait();
    ptx::dep_trigger();
    const uint32_t warps = blockDim.x >> 5;
    const uint32_t wid = blockIdx.x * warps + (threadIdx.x >> 5), nw = gridDim.x * warps;
    constexpr int UNROLL = 2;
    RecPackedItem<NIB_A, UNROLL> da;
    RecPackedItem<NIB_W, UNROLL> dw;
    const uint32_t steps = rec_steps(j.a, UNROLL), items_a = (uint32_t)j.a.panels * (REC_ROWS / 8) * steps;
    const uint32_t ww = after_items(wid, nw, items_a);
    rec_fetch<NIB_A, UNROLL>(j.pa, wid, steps, items_a, da);
    rec_fetch<NIB_W, UNROLL>(j.pw, ww, steps, (uint32_t)j.w.panels * (REC_ROWS / 8) * steps, dw);
    rec_decode_body<NIB_A, UNROLL>(j.pa, j.a, wid, nw, da);
    rec_decode_body<NIB_W, UNROLL>(j.pw, j.w, ww, nw, dw);
}

}  // namespace mx
