// Tensor-core form of the D <= 3 softmin sweep at float32 accuracy.
//
// The whole exponent of a pair,
//   v_ij = s xt_i . yt_j + H_j - m_i,   H_j = s (eps log w_j + pot_j - |yt_j|^2 / 2),
// is one dot product of length K = 32 between a row vector and a column
// vector of BF16 values, computed by tcgen05.mma with FP32 accumulation in
// tensor memory, so that the CUDA cores only evaluate ex2 and the sum.  Every
// float operand is split into three BF16 pieces (h + m + l, about 24
// significant bits, i.e. float32 accuracy); per coordinate the six products
// that matter at that accuracy (h.h, h.m, m.h, h.l, l.h, m.m) take six K
// slots, so the three coordinates use 18 slots.  H_j - C goes in three slots
// against 1.0, and the row shift -(m_i - C), rounded to BF16, in one slot
// against 1.0; C is the largest row shift of the block, so that the folded
// terms are small for every pair that matters.  The finish adds back exactly
// the shift the accumulator applied, in double precision.
//
// One CTA (4 warps) owns a row block of at most 128 rows (one tensor-memory
// lane and thread per row); columns come in tiles of kN.  Column staging is software
// pipelined: the indices of tile t+2 and the point of tile t+1 are loaded
// while the tensor core multiplies tile t+1 and the CTA sums tile t.  The
// indices come from the block's kept ranges (copied into shared memory once
// per CTA): every kChunkTiles tiles the CTA writes the column index of each
// position of the next chunk into one of two shared buffers, each thread
// kPerThr consecutive positions after one binary search.  Every wait is
// bounded.  Split blocks write partial sums; the CTA that completes a
// block's last item sums them in item order and finishes the rows.
#include <cfloat>
#include <cmath>

#include <cuda_bf16.h>

#include "otgb_internal.cuh"
#include "tcgen05.cuh"
#include "tile3.cuh"
#include "xtile.cuh"

namespace otgb {
namespace {

// Four CTAs of 128 threads share an SM (128 tensor-memory columns each): staging, MMA and sums of a tile follow each
// other within a CTA, and the CTAs fill each other's gaps.  Measured on the track-density workload (100k voxels per
// side): 128-column tiles, four CTAs 6.3e12 pairs/s; three CTAs 5.8e12; 256-column tiles, 256 threads, two CTAs 5.3e12;
// 64-column tiles, four CTAs 5.3e12.  Earlier forms: two accumulators per CTA 4.4-4.6e12; warp-specialised roles 4.6e12.
// Bound: the MUFU ex2 unit, 32 per clock per SM (1.0e13 pairs/s).  With MAXP (maximum and shift per pair besides)
// 5.8e12 pairs/s on 100k x 100k; otgb_softmin there 7.0 -> 1.9 ms against the two sweeps of softmin3_kernel, and
// 1000 x 800 109 -> 49 us (columns split over items, four launches, no host copies).
constexpr int kM = 128, kN = 128, kK = 32, kThreads = 128;
constexpr int kATile = kM * kK * 2;  // 8 KiB
constexpr int kBTile = kN * kK * 2;
constexpr uint32_t kTmemCols = kN;
// range entries of a block staged in shared memory; a block with more reads them from global memory
constexpr int kRngSmem = 1024;
// positions per expansion chunk (two buffers in flight) and per thread of an expansion
constexpr int kChunkTiles = 16, kChunk = kChunkTiles * kN, kPerThr = kChunk / kThreads;
static_assert(kPerThr * kThreads == kChunk && kPerThr % 4 == 0, "an expansion writes whole int4 groups");

// Word of position q (of a chunk) in the index buffer: 16-byte groups of four positions, group g stored at
// g ^ ((g >> 2) & 7) (a permutation of each aligned run of eight groups), so that both the expansion's
// 16-byte stores (a thread writes 16 consecutive positions) and the staging reads (a warp reads 32
// consecutive positions) are free of bank conflicts.
__device__ __forceinline__ int idx_word(int q) {
    const int g = q >> 2;
    return ((g ^ ((g >> 2) & 7)) << 2) | (q & 3);
}

// Column index of positions p0 .. p0 + kPerThr - 1 (those below `end`) from one block's range entries
// r[0 .. n) (the sentinel last, its position above every position asked for): a binary search for the
// first, then a forward walk.
template <typename Entries>
__device__ __forceinline__ void expand_positions(const Entries &r, int n, int p0, int end, int (&v)[kPerThr]) {
    int lo = 0, hi = n - 2;  // the last real entry
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (r(mid).y <= p0) lo = mid;
        else hi = mid - 1;
    }
    int k = lo;
    int2 cur = r(k), nxt = r(k + 1);
#pragma unroll
    for (int i = 0; i < kPerThr; ++i) {
        const int pq = p0 + i;
        v[i] = 0;
        if (pq < end) {
            while (nxt.y <= pq && k + 2 < n) {
                ++k;
                cur = nxt;
                nxt = r(k + 1);
            }
            v[i] = cur.x + (pq - cur.y);
        }
    }
}

struct Tc3Smem {
    unsigned char a[kATile];
    unsigned char b[kBTile];
    float red[4][8];
    int bc[2];
    unsigned long long mbar;
    uint32_t tslot;
    int2 rng[kRngSmem];
    alignas(16) int idx[2][kChunk];
};

using t3::bf2;
using t3::bfbits;
using t3::bfval;
using t3::hi_val;
using t3::kOne;
using t3::lo_val;
using t3::off32;
using t3::pk;
using t3::sdesc32;
using t3::split3x2;

// Scalar split for the row operand (once per CTA): v ~ h + m + l in BF16 (about 24 significant bits).  The per-tile
// column operand uses the packed form (t3::split3x2).  (Rounding with integer operations instead, which also frees the
// MUFU unit, measured 2 % slower: it costs issue slots.)
__device__ __forceinline__ void split3(float v, uint16_t &h, uint16_t &m, uint16_t &l) { xt::split3(v, 0.f, h, m, l); }

constexpr float kNoTerm = -1e29f;  // shift of a row without terms (absent columns have an exponent of about -1e30)

// MAXP: the shift is not known (no old value, or one that is no estimate of the result).  The accumulator then holds the
// pair's whole exponent (tile3.cuh) and the row keeps a running shift (xt::sum_row_max).
template <bool MAXP>
__global__ void __launch_bounds__(kThreads, 4) softmin3_tc_kernel(const __grid_constant__ SoftminLaunch L) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    Tc3Smem &S = *reinterpret_cast<Tc3Smem *>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int t = tid;  // row (tensor-memory lane)
    const int it = blockIdx.x;
    int4 item = L.items[it];
    OTGB_DCLAMP(item.x, 0, L.n_inst);
    const SoftminInst &I = L.inst[item.x];
    const int blk = item.y;
    int r0 = I.blk_row0[blk], r1 = I.blk_row0[blk + 1];
    OTGB_DCLAMP(r0, 0, I.n_rows + 1);
    OTGB_DCLAMP(r1, r0, min(I.n_rows, r0 + kM) + 1);
    const int nr = r1 - r0;
    const float eps = L.eps, s = L.s;
    const float4 *rows4 = reinterpret_cast<const float4 *>(I.rows);
    const float4 *cols4 = reinterpret_cast<const float4 *>(I.cols);

    // ---- the columns of this item: positions [cb, ce) of the block's kept columns; the block's
    // range entries (the sentinel last) into shared memory, visible after the first barrier below
    const int nkept = kept_cols(I, blk);
    int cb = item.z, ce = item.w;
    OTGB_DCLAMP(cb, 0, nkept + 1);
    OTGB_DCLAMP(ce, cb, nkept + 1);
    const int ncol = ce - cb;
    const int ntiles = (ncol + kN - 1) / kN;
    const bool ranged = I.col_rng != nullptr;
    const int nE = ranged ? I.rng_ptr[blk + 1] - I.rng_ptr[blk] : 0;
    const int2 *rb = ranged ? I.col_rng + I.rng_ptr[blk] : nullptr;
    const bool rng_local = ranged && nE <= kRngSmem;
    if (rng_local)
        for (int q = tid; q < nE; q += kThreads) S.rng[q] = rb[q];

    // ---- rows: centre of the block's bounding box, shifts, the row operand
    const bool valid = t < nr;
    float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
    if (valid) p = rows4[r0 + t];
    {
        float v[6] = {valid ? p.x : FLT_MAX, valid ? p.y : FLT_MAX, valid ? p.z : FLT_MAX,
                      valid ? -p.x : FLT_MAX, valid ? -p.y : FLT_MAX, valid ? -p.z : FLT_MAX};
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            for (int o = 16; o > 0; o >>= 1) v[q] = fminf(v[q], __shfl_xor_sync(0xffffffffu, v[q], o));
            if (lane == 0) S.red[warp][q] = v[q];
        }
    }
    if (tid == 0) {
        tc::mbar_init(&S.mbar, 1);
        tc::mbar_init_fence();
    }
    __syncthreads();
    // column index of every position of chunk ch (tiles ch * kChunkTiles ..) into S.idx[ch & 1]; the
    // sentinel's position (the block's number of kept columns) exceeds every position of the item
    auto expand = [&](int ch) {
        const int q0 = ch * kChunk + tid * kPerThr;  // item-relative position of this thread's first
        if (!ranged || q0 >= ncol) return;
        int v[kPerThr];
        if (rng_local) expand_positions([&](int k) { return S.rng[k]; }, nE, cb + q0, ce, v);
        else expand_positions([&](int k) { return rb[k]; }, nE, cb + q0, ce, v);
#pragma unroll
        for (int i = 0; i < kPerThr / 4; ++i)
            *reinterpret_cast<int4 *>(&S.idx[ch & 1][idx_word(tid * kPerThr + 4 * i)]) =
                make_int4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    };
    expand(0);  // read after the barriers of the row setup
    float c[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float lo = fminf(fminf(S.red[0][d], S.red[1][d]), fminf(S.red[2][d], S.red[3][d]));
        const float nhi = fminf(fminf(S.red[0][d + 3], S.red[1][d + 3]), fminf(S.red[2][d + 3], S.red[3][d + 3]));
        c[d] = 0.5f * (lo - nhi);
    }
    const float x0 = valid ? p.x - c[0] : 0.f, x1 = valid ? p.y - c[1] : 0.f, x2 = valid ? p.z - c[2] : 0.f;
    const double hx = 0.5 * ((double)x0 * x0 + (double)x1 * x1 + (double)x2 * x2);
    const bool far_row = MAXP && valid && hx > 0.5 * (double)xt::kFarRow / (double)s;
    float m = -INFINITY;
    if (!MAXP && valid) m = (float)((double)s * (hx - (double)I.row_old[r0 + t] / (double)I.lam));
    float Cb = 0.f;
    if constexpr (!MAXP) {
        float mx = m;
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0) S.red[warp][6] = mx;
        __syncthreads();
        Cb = fmaxf(fmaxf(S.red[0][6], S.red[1][6]), fmaxf(S.red[2][6], S.red[3][6]));
        if (!(Cb > -INFINITY)) Cb = 0.f;
    }
    const uint16_t mb = !MAXP && valid ? bfbits(-(m - Cb)) : (uint16_t)0;
    const double m_eff = (double)Cb - (double)bfval(mb);  // the shift the accumulator applies
    {
        uint32_t w[16];
        if constexpr (MAXP) {
            t3::row_words(x0, x1, x2, s, w);
        } else {
            uint16_t h[3], md[3], l[3];
            split3(s * x0, h[0], md[0], l[0]);
            split3(s * x1, h[1], md[1], l[1]);
            split3(s * x2, h[2], md[2], l[2]);
            // slots 6d .. 6d+5: h h m h l m (against the column's h m h l h m)
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const int b0 = 3 * d;  // three words per coordinate
                w[b0] = pk(h[d], h[d]);
                w[b0 + 1] = pk(md[d], h[d]);
                w[b0 + 2] = pk(l[d], md[d]);
            }
            w[9] = pk(kOne, kOne);  // slots 18, 19: against H pieces 1, 2
            w[10] = pk(kOne, mb);   // slot 20: H piece 3; slot 21: the shift
#pragma unroll
            for (int q = 11; q < 16; ++q) w[q] = 0u;
        }
        t3::store_words(S.a, t, w);
    }

    // ---- column staging: thread tid stages column tid of each tile
    auto load_idx = [&](int tile) -> int {
        const int pp = tile * kN + tid;
        int jj = -1;
        if (tile < ntiles && pp < ncol) {
            jj = ranged ? S.idx[(tile / kChunkTiles) & 1][idx_word((tile % kChunkTiles) * kN + tid)] : cb + pp;
            OTGB_DCLAMP(jj, 0, I.n_cols);
        }
        return jj;
    };
    int jc = -1, jn = -1;
    float4 rq = make_float4(0.f, 0.f, 0.f, 0.f);
    float rpot = 0.f;
    auto load_raw = [&]() {
        if (jc >= 0) {
            rq = cols4[jc];
            rpot = I.col_pot[jc];
        }
    };
    auto convert = [&]() {
        const bool okc = jc >= 0;
        const float y0 = okc ? rq.x - c[0] : 0.f, y1 = okc ? rq.y - c[1] : 0.f, y2 = okc ? rq.z - c[2] : 0.f;
        uint32_t w[16];
        if constexpr (MAXP) {
            t3::col_words(y0, y1, y2, rq.w, rpot, s, eps, okc, w);
        } else {
            const float sq = y0 * y0 + y1 * y1 + y2 * y2;
            float H = okc ? s * (fmaf(eps, rq.w, rpot) - 0.5f * sq) - Cb : -1e30f;
            if (H <= -1e30f) H = -1e30f;  // zero weight (log w = -inf); NaN goes on
            uint32_t H01, M01, L01, H2h, M2h, L2h;
            split3x2(y0, y1, H01, M01, L01);
            split3x2(y2, H, H2h, M2h, L2h);
            const uint16_t h[3] = {(uint16_t)(H01 >> 16), (uint16_t)H01, (uint16_t)(H2h >> 16)};
            const uint16_t md[3] = {(uint16_t)(M01 >> 16), (uint16_t)M01, (uint16_t)(M2h >> 16)};
            const uint16_t l[3] = {(uint16_t)(L01 >> 16), (uint16_t)L01, (uint16_t)(L2h >> 16)};
            const uint16_t hh[3] = {(uint16_t)H2h, (uint16_t)M2h, (uint16_t)L2h};
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const int b0 = 3 * d;
                w[b0] = pk(h[d], md[d]);
                w[b0 + 1] = pk(h[d], l[d]);
                w[b0 + 2] = pk(h[d], md[d]);
            }
            w[9] = pk(hh[0], hh[1]);
            w[10] = pk(hh[2], kOne);
#pragma unroll
            for (int q = 11; q < 16; ++q) w[q] = 0u;
        }
        t3::store_words(S.b, tid, w);
    };

    if (warp == 0) tc::tmem_alloc(&S.tslot, kTmemCols);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = S.tslot;
    float tot = 0.f, sh = kNoTerm;
    bool ok = true;
    // rows of this warp that exist: the epilogue of an empty warp is skipped
    const bool warp_rows = warp * 32 < nr;
    const uint32_t lanes = tmem + ((uint32_t)(warp * 32) << 16);
    jc = load_idx(0);
    load_raw();
    jn = load_idx(1);
    for (int tt = 0; tt < ntiles; ++tt) {
        convert();  // from registers
        jc = jn;
        load_raw();  // tile tt + 1
        jn = load_idx(tt + 2);
        tc::fence_proxy_async();
        tc::fence_before();
        __syncthreads();
        tc::fence_after();
        if (tid == 0) t3::issue(tmem, tc::smem_u32(S.a), tc::smem_u32(S.b), &S.mbar);
        // chunk c + 1 in the first iteration of chunk c, while the tensor core works: the index of tile T is read in
        // iteration T - 2, so the last read of chunk c - 1 (same buffer) came two iterations before, and the first read
        // of chunk c + 1 comes kChunkTiles - 2 iterations later, past this iteration's closing barrier
        if (tt % kChunkTiles == 0 && tt + kChunkTiles < ntiles) expand(tt / kChunkTiles + 1);
        if (!tc::mbar_wait(&S.mbar, (uint32_t)(tt & 1))) ok = false;
        ok = __all_sync(0xffffffffu, ok);  // tcgen05.ld below is warp-collective
        tc::fence_after();
        if (ok && warp_rows) {
            if constexpr (MAXP) xt::sum_row_max(lanes, tot, sh, [] {});
            else tot = xt::sum_row(lanes, tot, [] {});
        }
        tc::fence_before();
        __syncthreads();  // the operand tile and the accumulator are free again
    }
    ok = __syncthreads_and(ok) != 0;
    if (!ok && tid == 0 && L.tc_err) atomicOr(L.tc_err, 1u);
    tc::fence_after();
    if (warp == 0) tc::tmem_dealloc(tmem, kTmemCols);
    if (!ok) return;  // uniform
    if (tid == 0 && L.pairs) atomicAdd(L.pairs, (unsigned long long)nr * (unsigned long long)ncol);

    if (L.part) {
        // split block: partial sums (MAXP: with their shifts); the CTA that completes the block's last item combines
        // them in item order
        float2 *part2 = reinterpret_cast<float2 *>(L.part);
        if constexpr (MAXP) part2[(size_t)it * kPartRows + t] = make_float2(sh, tot);
        else L.part[(size_t)it * kPartRows + t] = tot;
        __threadfence();
        __syncthreads();
        if (tid == 0) {
            int fi = L.item_fin[it];
            OTGB_DCLAMP(fi, 0, L.n_fin);
            S.bc[0] = fi;
            S.bc[1] = atomicAdd(L.fin_count + fi, 1) + 1;
        }
        __syncthreads();
        const int4 fe = L.fin[S.bc[0]];
        if (S.bc[1] != fe.w) return;  // uniform
        __threadfence();
        tot = 0.f;
        if constexpr (MAXP) {
            const float2 *p = part2 + (size_t)fe.z * kPartRows + t;
            sh = kNoTerm;
            for (int q = 0; q < fe.w; ++q) sh = fmaxf(sh, __ldcg(&p[(size_t)q * kPartRows]).x);
            for (int q = 0; q < fe.w; ++q) {
                const float2 v = __ldcg(&p[(size_t)q * kPartRows]);
                tot += v.y * xt::ex2(v.x - sh);
            }
        } else {
            for (int q = 0; q < fe.w; ++q) {
                int iq = fe.z + q;
                OTGB_DCLAMP(iq, 0, L.n_items);
                tot += __ldcg(L.part + (size_t)iq * kPartRows + t);
            }
        }
    }
    float dmax = 0.f;
    if (valid) {
        const int r = r0 + t;
        if (!(tot >= 0x1p-60f && tot <= 0x1p60f) || far_row) {
            const int k = atomicAdd(L.n_fallback, 1);
            if (k < L.fallback_cap) L.fallback[k] = make_int4(item.x, r, blk, 0);
        } else {
            const double L2 = (MAXP ? (double)sh : m_eff) + log2((double)tot);
            const double tilde = -(double)I.lam * (L.eps_ln2 * L2 - (MAXP ? 0.0 : hx));
            double nw = tilde;
            if (I.row_old) {
                const double old = (double)I.row_old[r];
                nw = old + (double)I.omega * (tilde - old);
                dmax = (float)(fabs(nw - old) / (double)L.eps);
            }
            I.row_out[r] = (float)nw;
        }
    }
    for (int o = 16; o > 0; o >>= 1) dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    if (lane == 0 && L.delta_max) atomicMax(L.delta_max, __float_as_uint(dmax));
}


}  // namespace

void softmin3_tc_launch(const SoftminLaunch &L, bool maxp, cudaStream_t st) {
    static PerDevice<int> attr;
    attr.get([] {
        OTGB_CUDA_TRY(cudaFuncSetAttribute(softmin3_tc_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)sizeof(Tc3Smem)));
        OTGB_CUDA_TRY(cudaFuncSetAttribute(softmin3_tc_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)sizeof(Tc3Smem)));
        return 1;
    });
    if (maxp) softmin3_tc_kernel<true><<<L.n_items, kThreads, sizeof(Tc3Smem), st>>>(L);
    else softmin3_tc_kernel<false><<<L.n_items, kThreads, sizeof(Tc3Smem), st>>>(L);
    OTGB_CHECK_LAUNCH();
}

}  // namespace otgb
