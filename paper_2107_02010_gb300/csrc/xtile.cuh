// Tiles of the high-dimensional tensor-core kernels: the exponent of every (row, column) pair of a tile of 128
// rows x 128 columns as one contraction of K BF16 slots on the tensor cores, FP32 accumulation in tensor memory.
//
// Operands are split into NP BF16 pieces, v ~ h + m (+ l): NP = 2 keeps about 16 significant bits (products hh,
// hm, mh), NP = 3 about 24 (hh, hm, mh, mm, hl, lh), which is float32 accuracy.  The products run smallest first:
// the accumulator rounds at the size of what it holds, so only the hh steps round at full size.  Largest first
// would round at full size in every one of the six products.
//
// The columns' pieces lie in shared memory (canonical K-major layout without swizzle: core matrices of 8 columns x
// 16 bytes, contiguous along K, 8-column groups K x 16 bytes apart).  The rows' pieces lie in TENSOR MEMORY
// (tensor-memory lane = row, two consecutive K slots per 32-bit column): each thread owns one row, so it writes
// its operand with tcgen05.st without any transposition, and an MMA reads only its column operand through the
// shared-memory port (4 KB per 64 tensor clocks instead of 8 KB, which at 128 bytes per clock would saturate it
// and leave nothing for the arriving tiles).  Beside a 128-column accumulator the row pieces need NP K / 2
// columns, at most 96, so that two CTAs share an SM's 512 columns: one runs its MMAs while the other sums.
//
// The last K slots carry what the exponent adds to the cross term:
//   NP = 3: slot K-2: column H_j (its three pieces) against row 1; slot K-1: column 1 against row R_i (three pieces).
//   NP = 2: slots K-4, K-3: column (H1 | H2), (H3) against row 1, 1; slots K-2, K-1: column 1, 1 against row
//           (R1 | R2), (R3): three pieces of each although an operand has only two.
#pragma once

#include <cuda_bf16.h>

#include "tcgen05.cuh"

namespace otgb {
namespace xt {

constexpr int kRows = 128, kCols = 128;
// Rows with T = s |x - c|^2 above this (c: the centre of the row's block) are left to the safe kernel by the forms with a
// running shift.  A pair near such a row is a difference of numbers as large as T, rounded at 64 binades and more; a shift
// from old values shows that by a sum out of range, a running shift follows the wrong maximum (one row at 1e5 among points
// at 0 to 4, eps 0.09: every row of its block off by 70 to 150).
constexpr float kFarRow = 0x1p30f;
constexpr uint32_t kTmemCols = 256;  // accumulator (128) and the row operand(s)

// K slots of a point of D4 coordinates: the coordinates and the four (NP = 2) or two (NP = 3) folded slots, rounded
// up to whole MMA steps.  D4 is a multiple of 4, so both round to the same K.
__host__ __device__ constexpr int k_slots(int D4) { return (D4 + 4 + 15) / 16 * 16; }
__host__ __device__ constexpr int piece_bytes(int K) { return kCols * K * 2; }
__host__ __device__ constexpr int tile_bytes(int NP, int K) { return NP * piece_bytes(K); }

// byte offset of slot k of column c inside a piece
__host__ __device__ constexpr int off(int K, int c, int k) {
    return (c >> 3) * (K * 16) + (k >> 3) * 128 + (c & 7) * 16 + (k & 7) * 2;
}

template <int K> __device__ __forceinline__ uint64_t sdesc(uint32_t addr) {
    uint64_t d = (uint64_t)((addr & 0x3FFFF) >> 4);
    d |= (uint64_t)(128 >> 4) << 16;     // K-direction core-matrix stride
    d |= (uint64_t)(K * 16 >> 4) << 32;  // 8-column group stride
    d |= (uint64_t)1 << 46;              // descriptor version for this architecture
    return d;
}

constexpr uint16_t kOne = 0x3F80;  // 1.0 in BF16

__device__ __forceinline__ uint32_t pk(uint16_t lo, uint16_t hi) { return (uint32_t)lo | ((uint32_t)hi << 16); }
__device__ __forceinline__ uint16_t bfbits(float v) { return __bfloat16_as_ushort(__float2bfloat16_rn(v)); }
__device__ __forceinline__ float bfval(uint16_t b) { return __uint_as_float((uint32_t)b << 16); }

// v + rest ~ h + m + l in BF16 (26 bits of the sum: `rest` is what v lost to its own rounding)
__device__ __forceinline__ void split3(float v, float rest, uint16_t &h, uint16_t &m, uint16_t &l) {
    h = bfbits(v);
    const float r = v - bfval(h);
    m = bfbits(r);
    l = bfbits((r - bfval(m)) + rest);
}

// Two values rounded to BF16 by one packed conversion (its own pipe, not the MUFU unit's): `hi` in the high half,
// `lo` in the low half, each to nearest even as the scalar conversion rounds.
__device__ __forceinline__ uint32_t bf2(float hi, float lo) {
    uint32_t d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}
__device__ __forceinline__ float hi_val(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }
__device__ __forceinline__ float lo_val(uint32_t w) { return __uint_as_float(w << 16); }

// the NP pieces of two consecutive slots (k in the low half); rest0, rest1: what the values lost to their own rounding
// (they reach the third piece)
template <int NP, bool REST = false>
__device__ __forceinline__ void split2(float v0, float v1, uint32_t (&p)[NP], float rest0 = 0.f, float rest1 = 0.f) {
    p[0] = bf2(v1, v0);
    float r0 = v0 - lo_val(p[0]), r1 = v1 - hi_val(p[0]);
#pragma unroll
    for (int q = 1; q < NP; ++q) {
        if (REST && q == 2) {
            r0 += rest0;
            r1 += rest1;
        }
        p[q] = bf2(r1, r0);
        r0 -= lo_val(p[q]);
        r1 -= hi_val(p[q]);
    }
}

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// ---- tensor-memory stores and MMAs with the row operand in tensor memory
__device__ __forceinline__ void st8(uint32_t taddr, const uint32_t (&v)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(v[0]),
                 "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}
__device__ __forceinline__ void st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t db, uint32_t idesc, uint32_t acc) {
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(d),
                 "r"(a), "l"(db), "r"(idesc), "r"(acc));
}

// One tile's products (issued by one thread): row pieces at tensor-memory column `a`, column pieces at shared
// address `b`, accumulator `d` (overwritten).
// The tensor cores cut the running sum off towards zero after every step, so each step leaves a bias of half a unit
// in the last place against the sign of what the accumulator holds.  For a pair that matters the cross term is
// about T = s |x - c|^2 and H + R about -T: the K step with the folded slots goes in the middle, so that the sum
// passes through about T / 2 and -T / 2 instead of T, and `parity` 0 / 1 moves it by one step where the number of steps
// is even, so that the biases of even and odd tiles have opposite signs.  Where T is small beside the exponents (row
// blocks much smaller than the blur: single-scale solves, above all at the first scales of the schedule) the partial cross
// terms are what is small: with the folded step last (kFoldLast) a single step is cut off at the size of the exponent.  In
// the middle the same loss in every step stayed in the slowly contracting modes of f and g (single-scale solve, 60-D,
// reach 20: f off by 2.5e-7, CUDA cores 1.3e-7; now 1.4e-7; 48-D 1.7e-7, 1.3e-7, now 1.1e-7).  Cluster tiles stay with the
// middle: T is that of a whole cluster there, and the bundle means of a step are nearer to FP64 with it (2.8e-6 against
// 4.3e-6 last and 4.5e-6 on the CUDA cores at sigma 4).
constexpr int kFoldLast = 2;
constexpr float kFoldT = 4.f;
template <int NP, int K, int PAR> __device__ __forceinline__ void issue_as(uint32_t d, uint32_t a, uint32_t b) {
    constexpr uint32_t idesc = tc::idesc_bf16(kRows, kCols);
    constexpr int kP = NP == 3 ? 6 : 3, kS = K / 16;
    // (row piece, column piece), smallest products first
    constexpr int rp[6] = {NP == 3 ? 2 : 1, 0, NP == 3 ? 1 : 0, 1, 0, 0};
    constexpr int cp[6] = {0, NP == 3 ? 2 : 1, NP == 3 ? 1 : 0, 0, 1, 0};
    constexpr int fold = PAR == kFoldLast ? kS - 1 : (kS - 1 + PAR) / 2;  // place of the folded step
    uint32_t acc = 0u;
#pragma unroll
    for (int q = 0; q < kP; ++q)
#pragma unroll
        for (int k = 0; k < kS; ++k) {
            const int kk = k == fold ? kS - 1 : (k < fold ? k : k - 1);
            mma_ts(d, a + (uint32_t)(rp[q] * (K / 2) + kk * 8),
                   sdesc<K>(b + (uint32_t)(cp[q] * piece_bytes(K) + kk * 256)), idesc, acc);
            acc = 1u;
        }
}
template <int NP, int K> __device__ __forceinline__ void issue(uint32_t d, uint32_t a, uint32_t b, int parity) {
    if (parity == kFoldLast) issue_as<NP, K, kFoldLast>(d, a, b);
    else if (parity) issue_as<NP, K, 1>(d, a, b);
    else issue_as<NP, K, 0>(d, a, b);
}

// The row operand of this thread's row for centre c: s (x - c) in NP pieces, the folded slots, R = -s |x - c|^2 / 2
// - (M + Mlo).  `a`: tensor-memory column of the row pieces, with the warp's lane quadrant.  Returns T = s |x - c|^2 (0 when
// not valid).  Warp-collective.
template <int NP, int K>
__device__ __forceinline__ float stage_row(const float (&x)[K - 4], int D4, const float *c, float s, float M, bool valid,
                                          uint32_t a, float Mlo = 0.f) {
    const float4 *c4 = reinterpret_cast<const float4 *>(c);
    float T = 0.f;
    float4 sq = make_float4(0.f, 0.f, 0.f, 0.f);  // four short chains: less rounding than one long one
#pragma unroll
    for (int kk = 0; kk < K / 16; ++kk) {
        float v[16], d1[16];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int k4 = 4 * kk + q;
            float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
            if (4 * k4 < K - 4 && 4 * k4 < D4) {  // at most K - 4 coordinates
                const float4 cc = c4[k4];
                d = make_float4(x[4 * k4] - cc.x, x[4 * k4 + 1] - cc.y, x[4 * k4 + 2] - cc.z, x[4 * k4 + 3] - cc.w);
            }
            sq.x = fmaf(d.x, d.x, sq.x);
            sq.y = fmaf(d.y, d.y, sq.y);
            sq.z = fmaf(d.z, d.z, sq.z);
            sq.w = fmaf(d.w, d.w, sq.w);
            v[4 * q] = s * d.x;
            v[4 * q + 1] = s * d.y;
            v[4 * q + 2] = s * d.z;
            v[4 * q + 3] = s * d.w;
            d1[4 * q] = d.x;
            d1[4 * q + 1] = d.y;
            d1[4 * q + 2] = d.z;
            d1[4 * q + 3] = d.w;
        }
        uint32_t w[NP][8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            uint32_t p[NP];
            // Up to 12 coordinates with the rounding of s (x - c), which is the same error in every pair of the row (rms error of
            // otgb_softmin in 4 dimensions 0.95 -> 0.72 of the CUDA cores'); among more coordinates it averages (no difference
            // from 24 on).
            if constexpr (K == 16)
                split2<NP, true>(v[2 * j], v[2 * j + 1], p, fmaf(s, d1[2 * j], -v[2 * j]), fmaf(s, d1[2 * j + 1], -v[2 * j + 1]));
            else
                split2<NP>(v[2 * j], v[2 * j + 1], p);
#pragma unroll
            for (int q = 0; q < NP; ++q) w[q][j] = p[q];
        }
        if (kk == K / 16 - 1) {
            // R = P - M with what the product and the difference lose to rounding (where the finish adds M back its
            // own rounding cancels and Mlo is 0)
            const float hq = 0.5f * ((sq.x + sq.y) + (sq.z + sq.w)), P = -s * hq;
            if (valid) T = -2.f * P;
            const float R = P - M, bb = P - R;  // two-difference (Knuth)
            const float rest = (fmaf(-s, hq, -P) + ((P - (R + bb)) + (bb - M))) - Mlo;
            uint16_t r1, r2, r3;
            split3(valid ? R : 0.f, valid ? rest : 0.f, r1, r2, r3);
            if constexpr (NP == 3) {
                w[0][7] = pk(kOne, r1);
                w[1][7] = pk(0, r2);
                w[2][7] = pk(0, r3);
            } else {
                w[0][6] = pk(kOne, kOne);
                w[0][7] = pk(r1, r3);
                w[1][6] = 0u;
                w[1][7] = pk(r2, 0);
            }
        }
#pragma unroll
        for (int q = 0; q < NP; ++q) st8(a + (uint32_t)(q * (K / 2) + kk * 8), w[q]);
    }
    return T;
}

// The largest T of a block from its four row warps: each warp's maximum (T is never negative: its bits order as it does).
__device__ __forceinline__ void put_t(float T, float *slot, int lane) {
    const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(T));
    if (lane == 0) *slot = __uint_as_float(m);
}
__device__ __forceinline__ bool fold_last(const volatile float *t) {
    return fmaxf(fmaxf(t[0], t[1]), fmaxf(t[2], t[3])) < kFoldT;
}

// Column c of a tile: the point y centred at `cen` in NP pieces into `dst` (and `dst2` when non-null); the folded
// H slots are left 0 (put_h writes them), the ones are set.  Returns |y - cen|^2 / 2, summed in Acc: double where a
// tile is built once per solve, float (four short chains) where it is built per row block.
template <int NP, int K, class Acc>
__device__ __forceinline__ float build_col(const float *y, const float *cen, int D4, bool ok, int c, unsigned char *dst,
                                           unsigned char *dst2) {
    const float4 *y4 = reinterpret_cast<const float4 *>(y), *c4 = reinterpret_cast<const float4 *>(cen);
    Acc s0 = 0, s1 = 0, s2 = 0, s3 = 0;
#pragma unroll
    for (int ch = 0; ch < K / 8; ++ch) {
        uint32_t w[NP][4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
            if (8 * ch + 4 * h < K - 4 && ok && 8 * ch + 4 * h < D4) {
                const float4 u = y4[2 * ch + h], cc = c4[2 * ch + h];
                d = make_float4(u.x - cc.x, u.y - cc.y, u.z - cc.z, u.w - cc.w);
            }
            s0 += (Acc)d.x * d.x;
            s1 += (Acc)d.y * d.y;
            s2 += (Acc)d.z * d.z;
            s3 += (Acc)d.w * d.w;
            uint32_t p[NP], r[NP];
            split2<NP>(d.x, d.y, p);
            split2<NP>(d.z, d.w, r);
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                w[q][2 * h] = p[q];
                w[q][2 * h + 1] = r[q];
            }
        }
        if (ch == K / 8 - 1) {
            if constexpr (NP == 3) w[0][3] = pk(0, kOne);
            else w[0][3] = pk(kOne, kOne);
        }
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            const uint4 u = make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]);
            *reinterpret_cast<uint4 *>(dst + q * piece_bytes(K) + off(K, c, 8 * ch)) = u;
            if (dst2) *reinterpret_cast<uint4 *>(dst2 + q * piece_bytes(K) + off(K, c, 8 * ch)) = u;
        }
    }
    return (float)((Acc)0.5 * ((s0 + s1) + (s2 + s3)));
}

// H + rest of column c of a tile (three BF16 pieces)
template <int NP, int K> __device__ __forceinline__ void put_h(unsigned char *tile, int c, float H, float rest) {
    if (H <= -1e30f) {  // zero weight (log w = -inf) or past the end; NaN and +inf go on and make the row's sum NaN
        H = -1e30f;
        rest = 0.f;
    }
    uint16_t h1, h2, h3;
    split3(H, rest, h1, h2, h3);
    if constexpr (NP == 3) {
        *reinterpret_cast<uint32_t *>(tile + off(K, c, K - 2)) = pk(h1, kOne);
        *reinterpret_cast<uint32_t *>(tile + piece_bytes(K) + off(K, c, K - 2)) = pk(h2, 0);
        *reinterpret_cast<uint32_t *>(tile + 2 * piece_bytes(K) + off(K, c, K - 2)) = pk(h3, 0);
    } else {
        *reinterpret_cast<uint2 *>(tile + off(K, c, K - 4)) = make_uint2(pk(h1, h3), pk(kOne, kOne));
        *reinterpret_cast<uint2 *>(tile + piece_bytes(K) + off(K, c, K - 4)) = make_uint2(pk(h2, 0), 0u);
    }
}

// H = s (eps lw + pot - hn) with what its three roundings lose (products and sums with their exact errors)
template <int NP, int K>
__device__ __forceinline__ void put_h_sum(unsigned char *tile, int c, float s, float eps, float lw, float pot, float hn) {
    const float p = eps * lw, pe = fmaf(eps, lw, -p);
    const float a = p + pot, ab = a - p, ae = (p - (a - ab)) + (pot - ab);
    const float u = a - hn, ub = u - a, ue = (a - (u - ub)) - (hn + ub);
    const float H = s * u;
    put_h<NP, K>(tile, c, H, fmaf(s, u, -H) + s * ((pe + ae) + ue));
}

// ---- bulk copies and bounded waits
__device__ __forceinline__ void tma_load(void *dst, const void *src, uint32_t bytes, unsigned long long *bar) {
    const uint32_t b = tc::smem_u32(bar);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     tc::smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(b)
                 : "memory");
}
__device__ __forceinline__ void arrive(unsigned long long *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
}
// false when the phase did not complete within the limit or another role of the CTA gave up
__device__ __forceinline__ bool wait(unsigned long long *bar, uint32_t parity, const volatile int *abort) {
    const uint32_t addr = tc::smem_u32(bar);
    uint32_t done = 0;
    for (int it = 0; it < tc::kWaitLimit && !done; ++it) {
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(addr), "r"(parity)
            : "memory");
        if (!done && (it & 63) == 63 && *abort) return false;
    }
    return done != 0;
}

// sum of 2^v over one row of an accumulator of 128 columns at tensor-memory column `base` (with the warp's lane
// quadrant); the load of each 32 columns flies while the 32 before are summed.  freed() runs once the whole row is
// in registers (the accumulator may be overwritten from then on).
template <class F> __device__ __forceinline__ float sum_row(uint32_t base, float tot, F &&freed) {
    uint32_t va[32], vb[32];
    auto sum32 = [&](const uint32_t (&v)[32]) {
        float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
        for (int q = 0; q < 32; q += 4) {
            a0 += ex2(__uint_as_float(v[q]));
            a1 += ex2(__uint_as_float(v[q + 1]));
            a2 += ex2(__uint_as_float(v[q + 2]));
            a3 += ex2(__uint_as_float(v[q + 3]));
        }
        tot += (a0 + a1) + (a2 + a3);
    };
    tc::ld32_async(base, va);
    tc::ld_wait(va);
    tc::ld32_async(base + 32, vb);
    sum32(va);
    tc::ld_wait(vb);
    tc::ld32_async(base + 64, va);
    sum32(vb);
    tc::ld_wait(va);
    tc::ld32_async(base + 96, vb);
    sum32(va);
    tc::ld_wait(vb);
    freed();
    sum32(vb);
    return tot;
}

// The same without a known shift: the row's sum is tot 2^sh.  Per 32 columns the maximum; where it passes the shift by
// 30 binades the sum is rescaled to it (rare after the first columns, so the branch is cheap).
template <class F> __device__ __forceinline__ void sum_row_max(uint32_t base, float &tot, float &sh, F &&freed) {
    uint32_t va[32], vb[32];
    auto sum32 = [&](const uint32_t (&v)[32]) {
        float m0 = __uint_as_float(v[0]), m1 = __uint_as_float(v[1]);
#pragma unroll
        for (int q = 2; q < 32; q += 2) {
            m0 = fmaxf(m0, __uint_as_float(v[q]));
            m1 = fmaxf(m1, __uint_as_float(v[q + 1]));
        }
        m0 = fmaxf(m0, m1);
        if (m0 > sh + 30.f) {
            tot *= ex2(sh - m0);
            sh = m0;
        }
        float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
        for (int q = 0; q < 32; q += 4) {
            a0 += ex2(__uint_as_float(v[q]) - sh);
            a1 += ex2(__uint_as_float(v[q + 1]) - sh);
            a2 += ex2(__uint_as_float(v[q + 2]) - sh);
            a3 += ex2(__uint_as_float(v[q + 3]) - sh);
        }
        tot += (a0 + a1) + (a2 + a3);
    };
    tc::ld32_async(base, va);
    tc::ld_wait(va);
    tc::ld32_async(base + 32, vb);
    sum32(va);
    tc::ld_wait(vb);
    tc::ld32_async(base + 64, va);
    sum32(vb);
    tc::ld_wait(va);
    tc::ld32_async(base + 96, vb);
    sum32(va);
    tc::ld_wait(vb);
    freed();
    sum32(vb);
}

// ---- the cluster-tiled kernels: column tiles prepared in global memory, walked cluster by cluster
constexpr int kStageBudget = 96 * 1024;  // shared memory for column tiles: two CTAs per SM
constexpr int kMaxStages = 6;

template <int NP, int K> struct Geom {
    static constexpr int tile = tile_bytes(NP, K);
    static constexpr int st = kStageBudget / tile;
    static constexpr int stages = st > kMaxStages ? kMaxStages : st;
    // a second row operand where 256 tensor-memory columns hold it: the next cluster's rows are then staged while
    // the MMAs of the current one run
    static constexpr int abuf = kCols + 2 * NP * (K / 2) <= (int)kTmemCols ? 2 : 1;
    static_assert(kCols + NP * (K / 2) <= (int)kTmemCols && stages >= 2, "tile does not fit");
};

// Walks the tiles of the kept column clusters of a block in cluster order.
struct TileIt {
    int w = -1;
    unsigned u = 0u;
    int J = -1, g = 0, gend = 0;
};
__device__ __forceinline__ bool tile_next(TileIt &it, const unsigned *words, int nwords, const int *tile0) {
    if (it.g + 1 < it.gend) {
        ++it.g;
        return true;
    }
    for (;;) {
        while (it.u == 0u) {
            if (++it.w >= nwords) return false;
            it.u = words[it.w];
        }
        const int bit = __ffs(it.u) - 1;
        it.u &= it.u - 1u;
        it.J = it.w * 32 + bit;
        it.g = tile0[it.J];
        it.gend = tile0[it.J + 1];
        if (it.g < it.gend) return true;
    }
}

}  // namespace xt
}  // namespace otgb
