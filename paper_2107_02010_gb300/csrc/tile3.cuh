// Operands of the D <= 3 tensor-core tiles without a known row shift: K = 32 BF16 slots whose dot product is the whole
// base-2 exponent of a pair, -s |x - y|^2 / 2 + s (eps log w + pot), at float32 accuracy.
//
// Every float operand is split into three BF16 pieces (h + m + l); per coordinate the six products that matter take six
// slots.  The rows may come as the caller has them, so that |x - c| |y - c| (c the block's centre) is much larger than any
// exponent that matters; the slots are arranged so that each of the two K = 16 steps is small by itself for such a pair:
// step 0 holds coordinates 0 and 1 with their own share of the squares (two pieces of -s (y0^2 + y1^2) / 2 against 1, two
// of -s (x0^2 + x1^2) / 2), step 1 coordinate 2 and everything else (three pieces each).  The tensor cores cut the sum off
// towards zero after each step, at the size of what it holds.
#pragma once

#include "tcgen05.cuh"
#include "xtile.cuh"

namespace otgb {
namespace t3 {

constexpr int kTile = 128, kK = 32, kBytes = kTile * kK * 2;  // 8 KiB per operand of 128 rows or columns

// K-major canonical layout of a tile with 32 K-columns: 8-row x 16-byte core matrices, 4 along K (leading byte offset
// 128), 8-row groups 512 bytes apart
__device__ __forceinline__ int off32(int r, int k) { return (r >> 3) * 512 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2; }

__device__ __forceinline__ uint64_t sdesc32(uint32_t addr) {
    uint64_t d = (uint64_t)((addr & 0x3FFFF) >> 4);
    d |= (uint64_t)(128 >> 4) << 16;
    d |= (uint64_t)(512 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

using xt::bf2;
using xt::bfbits;
using xt::bfval;
using xt::hi_val;
using xt::kOne;
using xt::lo_val;
using xt::pk;

// Two values split at once: H, M, L hold the h, m, l pieces of a in their high halves and of b in their low halves.  The
// packed conversion rounds each half to nearest even, as the scalar one does; it runs on its own pipe, leaving the MUFU
// unit to ex2.  rest: what b lost to its own rounding.
__device__ __forceinline__ void split3x2(float a, float b, uint32_t &H, uint32_t &M, uint32_t &L, float rest = 0.f) {
    H = bf2(a, b);
    const float ra = a - hi_val(H), rb = b - lo_val(H);
    M = bf2(ra, rb);
    L = bf2(ra - hi_val(M), (rb - lo_val(M)) + rest);
}

// First word (two K slots) of coordinate d.
__device__ __forceinline__ constexpr int coord_word(int d) { return d == 2 ? 8 : 3 * d; }

// The row operand of centred point x: 16 words of two slots.
__device__ __forceinline__ void row_words(float x0, float x1, float x2, float s, uint32_t (&w)[16]) {
    const float x[3] = {s * x0, s * x1, s * x2};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        uint16_t h, m, l;
        xt::split3(x[d], 0.f, h, m, l);
        const int b0 = coord_word(d);  // h h m h l m (against the column's h m h l h m)
        w[b0] = pk(h, h);
        w[b0 + 1] = pk(m, h);
        w[b0 + 2] = pk(l, m);
    }
    const double R01 = -0.5 * (double)s * ((double)x0 * x0 + (double)x1 * x1);
    const uint16_t ra = bfbits((float)R01), rb = bfbits((float)(R01 - (double)bfval(ra)));
    const double R2 = (R01 - (double)bfval(ra) - (double)bfval(rb)) - 0.5 * (double)s * ((double)x2 * x2);
    uint16_t r1, r2, r3;
    xt::split3((float)R2, (float)(R2 - (double)(float)R2), r1, r2, r3);
    w[6] = pk(kOne, kOne);
    w[7] = pk(ra, rb);
    w[11] = pk(kOne, kOne);
    w[12] = pk(kOne, r1);
    w[13] = pk(r2, r3);
    w[14] = w[15] = 0u;
}

// The column operand of centred point y with log weight lw and potential pot; in = false: no column (exponent -1e30).
__device__ __forceinline__ void col_words(float y0, float y1, float y2, float lw, float pot, float s, float eps, bool in,
                                          uint32_t (&w)[16]) {
    // |y0|^2 + |y1|^2 with its rounding errors (Knuth's two-sum, products by FMA), times -s/2; two BF16 pieces of it stay
    // with those coordinates, what they leave joins the rest of H, which is summed with its errors too
    const float hs = -0.5f * s;
    const float p0 = y0 * y0, p1 = y1 * y1, t01 = p0 + p1, tb = t01 - p0;
    const float te = ((p0 - (t01 - tb)) + (p1 - tb)) + (fmaf(y0, y0, -p0) + fmaf(y1, y1, -p1));
    const float q01 = hs * t01, qe = fmaf(hs, t01, -q01) + hs * te;
    const uint32_t wa = bf2(0.f, q01);
    const float qa = q01 - lo_val(wa);
    const uint32_t wb = bf2(0.f, qa);
    const float rem = qa - lo_val(wb);
    w[6] = in ? pk((uint16_t)wa, (uint16_t)wb) : 0u;
    w[7] = pk(kOne, kOne);
    const float u = fmaf(eps, lw, pot), v = s * u, ve = fmaf(s, u, -v);
    const float z = y2 * y2, g = hs * z, ge = fmaf(hs, z, -g) + hs * fmaf(y2, y2, -z);
    const float S1 = v + g, sb = S1 - v, se = (v - (S1 - sb)) + (g - sb);
    float H = S1 + rem;
    const float hb = H - S1;
    float rest = ((S1 - (H - hb)) + (rem - hb)) + (se + (ve + ge) + qe);
    if (!in || H <= -1e30f) {  // absent, or zero weight (log w = -inf); NaN goes on
        H = -1e30f;
        rest = 0.f;
    }
    uint32_t H01, M01, L01, H2h, M2h, L2h;
    split3x2(y0, y1, H01, M01, L01);
    split3x2(y2, H, H2h, M2h, L2h, rest);
    const uint16_t h[3] = {(uint16_t)(H01 >> 16), (uint16_t)H01, (uint16_t)(H2h >> 16)};
    const uint16_t m[3] = {(uint16_t)(M01 >> 16), (uint16_t)M01, (uint16_t)(M2h >> 16)};
    const uint16_t l[3] = {(uint16_t)(L01 >> 16), (uint16_t)L01, (uint16_t)(L2h >> 16)};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int b0 = coord_word(d);
        w[b0] = pk(h[d], m[d]);
        w[b0 + 1] = pk(h[d], l[d]);
        w[b0 + 2] = pk(h[d], m[d]);
    }
    w[11] = pk((uint16_t)H2h, (uint16_t)M2h);
    w[12] = pk((uint16_t)L2h, kOne);
    w[13] = pk(kOne, kOne);
    w[14] = w[15] = 0u;
}

__device__ __forceinline__ void store_words(unsigned char *tile, int r, const uint32_t (&w)[16]) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
        *reinterpret_cast<uint4 *>(tile + off32(r, 8 * q)) = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
}

// acc[128 x 128] = A . B^T over the 32 slots, completion on `bar` (one thread)
__device__ __forceinline__ void issue(uint32_t acc, uint32_t a, uint32_t b, void *bar) {
#pragma unroll
    for (int kk = 0; kk < kK / 16; ++kk)
        tc::mma_bf16(acc, sdesc32(a + kk * 256), sdesc32(b + kk * 256), tc::idesc_bf16(kTile, kTile), kk > 0 ? 1u : 0u);
    tc::commit(bar);
}

}  // namespace t3
}  // namespace otgb
