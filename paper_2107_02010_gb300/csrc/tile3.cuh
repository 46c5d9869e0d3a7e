// Operands of the D <= 3 tensor-core tiles without a known row shift: K = 32 BF16 slots whose dot product is the whole
// base-2 exponent of a pair, -s |x - y|^2 / 2 + s (eps log w + pot), at float32 accuracy.
//
// Every float operand is split into three BF16 pieces (h + m + l); six products per coordinate matter (ml, lm and ll are
// below 2^-24 of hh).  The rows may come as the caller has them, so that |x - c| |y - c| (c the block's centre) and the
// squares are much larger than any exponent that matters, while their sum is small.  Two things keep that sum's error down:
//  - The row's pieces hold s (x - c) with what the product loses to rounding.  Without it (T 2^-25 for every pair of the
//    row, T = s |x - c| |y - c|) the error of a row is that of a single float product.
//  - A tensor-core step aligns its products and the accumulator to the largest of them and cuts off what lies some 24 bits
//    below, towards zero.  The first K = 16 step holds hh, hm, mh and the leading pieces of H and R, whose bits lie above
//    the cut for the larger coordinates; it leaves something small, to which the second step adds hl, mm, lh and the last
//    pieces of H and R (2^-16 of the others) without losing their bits.
// otgb_softmin, rms error against FP64, 3,000 x 2,500 points over 30 units in one / two / three dimensions, eps 1:
// 4.1e-7 / 4.5e-7 / 3.6e-7 (CUDA cores 1.3e-6 / 1.7e-6 / 1.4e-6; without the rounding of s (x - c) and coordinate by
// coordinate 1.8e-6 / 1.6e-6 / 0.9e-6; small products first 5.3e-7 / 5.4e-7 / 4.2e-7).
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

// Words (two K slots each) of one operand.  Slots 0-8: hh, hm, mh of the coordinates; 9, 10: H's leading pieces, 11, 12:
// R's; slots 16-24: hl, mm, lh; 25: H's last piece, 26: R's.
//
// The row operand of centred point x.
__device__ __forceinline__ void row_words(float x0, float x1, float x2, float s, uint32_t (&w)[16]) {
    const float x[3] = {s * x0, s * x1, s * x2};
    const float xr[3] = {fmaf(s, x0, -x[0]), fmaf(s, x1, -x[1]), fmaf(s, x2, -x[2])};
    uint16_t h[3], m[3], l[3], r1, r2, r3;
#pragma unroll
    for (int d = 0; d < 3; ++d) xt::split3(x[d], xr[d], h[d], m[d], l[d]);
    const double R = -0.5 * (double)s * ((double)x0 * x0 + (double)x1 * x1 + (double)x2 * x2);
    xt::split3((float)R, (float)(R - (double)(float)R), r1, r2, r3);
    w[0] = pk(h[0], h[0]); w[1] = pk(m[0], h[1]); w[2] = pk(h[1], m[1]); w[3] = pk(h[2], h[2]);
    w[4] = pk(m[2], kOne); w[5] = pk(kOne, r1); w[6] = pk(r2, 0);
    w[8] = pk(h[0], m[0]); w[9] = pk(l[0], h[1]); w[10] = pk(m[1], l[1]); w[11] = pk(h[2], m[2]);
    w[12] = pk(l[2], kOne); w[13] = pk(r3, 0);
    w[7] = w[14] = w[15] = 0u;
}

// The column operand of centred point y with log weight lw and potential pot; in = false: no column (exponent -1e30).
__device__ __forceinline__ void col_words(float y0, float y1, float y2, float lw, float pot, float s, float eps, bool in,
                                          uint32_t (&w)[16]) {
    // H = s (eps lw + pot) - s |y|^2 / 2 with its rounding errors (Knuth's two-sum, products by FMA)
    const float hs = -0.5f * s;
    const float p0 = y0 * y0, p1 = y1 * y1, t01 = p0 + p1, tb = t01 - p0;
    const float te = ((p0 - (t01 - tb)) + (p1 - tb)) + (fmaf(y0, y0, -p0) + fmaf(y1, y1, -p1));
    const float q01 = hs * t01, qe = fmaf(hs, t01, -q01) + hs * te;
    const float u = fmaf(eps, lw, pot), v = s * u, ve = fmaf(s, u, -v);
    const float z = y2 * y2, g = hs * z, ge = fmaf(hs, z, -g) + hs * fmaf(y2, y2, -z);
    const float S1 = v + g, sb = S1 - v, se = (v - (S1 - sb)) + (g - sb);
    float H = S1 + q01;
    const float hb = H - S1;
    float rest = ((S1 - (H - hb)) + (q01 - hb)) + (se + (ve + ge) + qe);
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
    w[0] = pk(h[0], m[0]); w[1] = pk(h[0], h[1]); w[2] = pk(m[1], h[1]); w[3] = pk(h[2], m[2]);
    w[4] = pk(h[2], (uint16_t)H2h); w[5] = pk((uint16_t)M2h, kOne); w[6] = pk(kOne, 0);
    w[8] = pk(l[0], m[0]); w[9] = pk(h[0], l[1]); w[10] = pk(m[1], h[1]); w[11] = pk(l[2], m[2]);
    w[12] = pk(h[2], (uint16_t)L2h); w[13] = pk(kOne, 0);
    w[7] = w[14] = w[15] = 0u;
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
