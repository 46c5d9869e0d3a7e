// Label transfer (Eq. (7)) for 3 < D, D4 <= 60 on the tensor cores:
//   Lab_il = sum_{j : l_j = l} b_j exp((f_i + g_j - |x_i - y_j|^2/2) / eps).
// The exponent of every pair is one tensor-core dot product of three-piece BF16 operands (xtile.cuh), the columns in
// tiles of 128 centred at their k-means cluster's centroid, as in softmin_tcc.cu; the row shift is M_i = -s f_i, so
// the accumulator holds the pair's base-2 exponent and a class sum needs no rescaling.
//
// Which pairs.  A float32 sum does not see a term below 2^-126: ex2.approx.ftz returns 0 there.  Rows and columns are
// grouped by the nearest of the column side's centroids, and a (row cluster, column cluster) pair whose largest
// possible exponent (from centroids, radii and the largest f and eps log b + g) is below 2^-130 is not visited: its
// terms are exact zeros in the dense sum as well.  With 20 separate fiber bundles that leaves one pair in twenty.
//
// The columns are sorted by (cluster, label).  A thread keeps one running sum and adds it to its row's score of the
// current class when the class changes: a mask of 128 bits per tile says where (none in most groups of 32 columns,
// which then take the plain sum).  Scores are kept class-major while they are summed, so that the 32 rows of a warp
// add to 32 consecutive floats; every row belongs to one thread, so the order of the additions is fixed.
//
// Near ties.  A row's label is a whole number and must not depend on which kernel summed its classes, so a row whose two
// best scores lie within kTie of each other is decided by the arithmetic of the CUDA-core kernel (transport_gen_kernel):
// the centre of the row's block in that kernel's k-means order, its FMA chains and its order of sums.  That costs the
// block order (a k-means over all rows) when there is such a row, and nothing otherwise.  Up to kFewTies rows take a CTA each;
// more of them (an atlas with two labels on the same fibers ties every row) that kernel itself, over the blocks and classes
// concerned: 60k x 50k fibers, two such labels, 262 ms with a CTA per row, 20.5 now (transport_gen_kernel alone 24.2, 20 now
// that its FMAs are packed); a small atlas of ties pays for the sweep that decided nothing (5,000 x 5,000: 1.3 ms, 1.0).
//
// Measured (60k x 50k fibers, 60-D, 20 labels that split every bundle; whole call): 24.5 -> 3.1 ms, of which the sweep
// 0.66 (13 % of the pairs visited; dense at the tensor bound: 1.2), the two k-means and their sorts 0.8, about 20 near
// ties 1.4 (the k-means over all rows 1.28, their sums 0.15).  transport_gen_kernel alone took 22 ms.  Error of the scores against FP64 8.1e-7 - 9.1e-7 -> 3.6e-7 - 7.1e-7.
#include <cmath>
#include <cstring>

#include "kmeans.cuh"
#include "prims.cuh"
#include "solver.cuh"
#include "transport.cuh"
#include "xtile.cuh"

namespace otgb {
namespace {

constexpr int kThreads = 192;
constexpr int kN = xt::kCols;
constexpr float kSkip = -130.f;  // base-2 exponents below this are 0 in float32 (2^-126 is the smallest normal number)

constexpr int kFewTies = 256;       // rows that a CTA each decides
// Two scores within this of each other (relative) are a near tie: four times the scores' error at eps 4 (at most 5e-6 against
// the CUDA-core kernel), and where the exponents are larger what they are rounded at there.  That kernel rounds s u_j (u_j =
// eps log b_j + g_j), its sum with -s |y - c|^2 / 2 and the product once each and sums the cross term over the coordinates: an
// exponent is off by up to about 3 2^-24 s |u| + 8 2^-24 s r^2 (r: the row cluster's radius), a score by ln 2 of that, the
// difference of two by twice as much: 2.5e-7 s |u| + 6.6e-7 s r^2.  A column that matters has u between -|f| and the largest u.
constexpr float kTie = 2e-5f, kTieRel = 5e-7f;

struct XferArgs {
    const float *rows;  // packed rows, grouped by cluster
    const float *f;
    int D4;
    const int *blk_row0, *blk_cl;
    const unsigned *bits;  // row cluster x nwords
    int nwords;
    unsigned char *tiles;
    const float *half_norm;
    const int *tile0, *tile_cl, *off;  // first tile of a cluster, cluster of a tile, first column of a cluster
    int ntiles;
    const float *ccen;
    const float *col_logw, *g;
    const int *lab;   // label per sorted column (L: ignored)
    int *tile_lab;    // label per tile column
    uint4 *tile_chg;  // per tile: bit q = column q has another label than column q - 1
    float *score;     // class-major, L x ld
    size_t ld;
    int L;
    float eps, s;
    unsigned *err;
};

struct Ctl {
    unsigned words[kTccMaxWords];
    unsigned long long full[xt::kMaxStages], empty[xt::kMaxStages], acc_full, acc_free, a_ready[2], drain;
    uint32_t tslot;
    int abort;
};

// H of every tile column, its label, and the label changes of the tile.
template <int K> __global__ void __launch_bounds__(kN) xfer_tiles_kernel(const __grid_constant__ XferArgs A) {
    const int g = blockIdx.x, c = threadIdx.x;
    const int J = A.tile_cl[g];
    const int end = A.off[J + 1], first = A.off[J] + (g - A.tile0[J]) * kN;
    const int j = first + c;
    float lw = -INFINITY, pot = 0.f;
    if (j < end) {
        lw = A.col_logw[j];
        pot = A.g[j];
    }
    xt::put_h_sum<3, K>(A.tiles + (size_t)g * xt::tile_bytes(3, K), c, A.s, A.eps, lw, pot, A.half_norm[(size_t)g * kN + c]);
    // past the cluster's end: the last label goes on (its terms are 0)
    const int l = A.lab[min(j, end - 1)], lp = c > 0 ? A.lab[min(j - 1, end - 1)] : l;
    A.tile_lab[(size_t)g * kN + c] = l;
    const unsigned w = __ballot_sync(0xffffffffu, l != lp);
    if ((c & 31) == 0) reinterpret_cast<unsigned *>(A.tile_chg + g)[c >> 5] = w;
}

// Largest f (rows) or eps log w + g (columns) of each cluster, one warp per cluster; NaN counts as +inf, so that the
// cluster is visited.
// top (optional; zero it first): the largest positive finite value over all of them, as its bits.
__global__ void xfer_max_kernel(const int *off, int ncl, const float *v, const float *lw, float eps, float *out, unsigned *top) {
    const int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (c >= ncl) return;
    float m = -INFINITY;
    for (int i = off[c] + lane; i < off[c + 1]; i += 32) {
        const float u = lw ? fmaf(eps, lw[i], v[i]) : v[i];
        m = u == u ? fmaxf(m, u) : INFINITY;
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) {
        out[c] = m;
        if (top && m > 0.f && m < INFINITY) atomicMax(top, __float_as_uint(m));
    }
}

// Keep bits of row cluster blockIdx.x.  !(bound < kSkip) keeps a pair whose bound is NaN.
__global__ void xfer_mask_kernel(const float *cr, const float *rr, const float *mr, const float *cc, const float *rc,
                                 const float *mc, int ncl, int D4, float s, unsigned *bits, int nwords) {
    __shared__ float cI[64];
    const int I = blockIdx.x;
    if (threadIdx.x < D4) cI[threadIdx.x] = cr[(size_t)I * D4 + threadIdx.x];
    __syncthreads();
    const float rI = rr[I], mI = mr[I];
    for (int base = 0; base < nwords * 32; base += blockDim.x) {
        const int J = base + threadIdx.x;
        bool keep = false;
        if (J < ncl) {
            const float4 *c4 = reinterpret_cast<const float4 *>(cc + (size_t)J * D4);
            float d2 = 0.f;
            for (int q = 0; q < D4 / 4; ++q) {
                const float4 v = c4[q];
                const float t0 = cI[4 * q] - v.x, t1 = cI[4 * q + 1] - v.y, t2 = cI[4 * q + 2] - v.z, t3 = cI[4 * q + 3] - v.w;
                d2 = fmaf(t0, t0, fmaf(t1, t1, fmaf(t2, t2, fmaf(t3, t3, d2))));
            }
            // a little less than the true gap: the distance is rounded, and the radii are
            const float gap = fmaxf(sqrtf(d2) * 0.99999f - rI - rc[J], 0.f);
            keep = !(s * (mI + mc[J] - 0.5f * gap * gap) < kSkip);
        }
        const unsigned w = __ballot_sync(0xffffffffu, keep);
        if ((threadIdx.x & 31) == 0 && (J >> 5) < nwords) bits[(size_t)I * nwords + (J >> 5)] = w;
    }
}

// One CTA per row block (at most 128 rows of one row cluster); the roles of softmin_tcc_kernel.
template <int K> __global__ void __launch_bounds__(kThreads, 2) xfer_kernel(const __grid_constant__ XferArgs A) {
    using G = xt::Geom<3, K>;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *tiles_s = smem_raw;
    Ctl &S = *reinterpret_cast<Ctl *>(smem_raw + G::stages * G::tile);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31, D4 = A.D4;
    const int r0 = A.blk_row0[blockIdx.x], nr = min(A.blk_row0[blockIdx.x + 1] - r0, xt::kRows);
    const float s = A.s;
    volatile int *abort = &S.abort;
    if (t == 0) {
        S.abort = 0;
        for (int q = 0; q < G::stages; ++q) {
            tc::mbar_init(&S.full[q], 1);
            tc::mbar_init(&S.empty[q], 1);
        }
        tc::mbar_init(&S.acc_full, 1);
        tc::mbar_init(&S.acc_free, 128);
        tc::mbar_init(&S.a_ready[0], 128);
        tc::mbar_init(&S.a_ready[1], 128);
        tc::mbar_init(&S.drain, 1);
        tc::mbar_init_fence();
    }
    if (warp == 5) tc::tmem_alloc(&S.tslot, xt::kTmemCols);
    const unsigned *bits = A.bits + (size_t)A.blk_cl[blockIdx.x] * A.nwords;
    for (int w = t; w < A.nwords; w += kThreads) S.words[w] = bits[w];
    const bool valid = t < nr;
    float Mi = 0.f, Mlo = 0.f;  // -s f in two floats
    float x[K - 4];
    if (warp < 4) {
        const float4 *xr4 = reinterpret_cast<const float4 *>(A.rows + (size_t)(r0 + (valid ? t : 0)) * D4);
#pragma unroll
        for (int q = 0; q < K / 4 - 1; ++q) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (valid && 4 * q < D4) v = xr4[q];
            x[4 * q] = v.x;
            x[4 * q + 1] = v.y;
            x[4 * q + 2] = v.z;
            x[4 * q + 3] = v.w;
        }
        if (valid) {
            const float f = A.f[r0 + t];
            Mi = __fmul_rn(-s, f);
            Mlo = fmaf(-s, f, -Mi);
        }
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = S.tslot;

    if (warp == 4) {
        if (lane == 0) {
            xt::TileIt it;
            int k = 0;
            while (xt::tile_next(it, S.words, A.nwords, A.tile0)) {
                const int st = k % G::stages;
                if (k >= G::stages && !xt::wait(&S.empty[st], (uint32_t)((k / G::stages - 1) & 1), abort)) {
                    *abort = 1;
                    break;
                }
                xt::tma_load(tiles_s + st * G::tile, A.tiles + (size_t)it.g * G::tile, (uint32_t)G::tile, &S.full[st]);
                ++k;
            }
            // nothing in flight at exit: the last copy into each stage has landed
            for (int q = max(0, k - G::stages); q < k; ++q)
                if (!tc::mbar_wait(&S.full[q % G::stages], (uint32_t)((q / G::stages) & 1))) *abort = 1;
        }
        __syncwarp();
    } else if (warp == 5) {
        if (lane == 0) {
            bool ok = true;
            xt::TileIt it;
            int k = 0, aJ = -1, na = 0;
            while (xt::tile_next(it, S.words, A.nwords, A.tile0)) {
                const int st = k % G::stages;
                if (it.J != aJ) {
                    if (!xt::wait(&S.a_ready[na % G::abuf], (uint32_t)((na / G::abuf) & 1), abort)) {
                        ok = false;
                        break;
                    }
                    aJ = it.J;
                    ++na;
                }
                if (!xt::wait(&S.full[st], (uint32_t)((k / G::stages) & 1), abort) ||
                    (k >= 1 && !xt::wait(&S.acc_free, (uint32_t)((k - 1) & 1), abort))) {
                    ok = false;
                    break;
                }
                tc::fence_after();
                xt::issue<3, K>(tmem, tmem + kN + (uint32_t)(((na - 1) % G::abuf) * 3 * (K / 2)),
                                tc::smem_u32(tiles_s + st * G::tile), k & 1);
                tc::commit(&S.empty[st]);
                tc::commit(&S.acc_full);
                ++k;
            }
            tc::commit(&S.drain);
            if (!tc::mbar_wait(&S.drain, 0)) ok = false;
            if (!ok) *abort = 1;
        }
        __syncwarp();
    } else {
        const uint32_t lanes = tmem + ((uint32_t)(warp * 32) << 16);
        int na = 0;
        auto stage = [&](int J) {
            const uint32_t a = lanes + kN + (uint32_t)((na % G::abuf) * 3 * (K / 2));
            xt::stage_row<3, K>(x, D4, A.ccen + (size_t)J * D4, s, Mi, valid, a, Mlo);
            xt::st_wait();
            tc::fence_before();
            xt::arrive(&S.a_ready[na % G::abuf]);
            ++na;
        };
        int cur = A.L;  // class of the running sum; L: ignored
        float tot = 0.f;
        float *mine = A.score + (r0 + t);
        auto flush = [&](int next) {
            if (valid && cur < A.L) atomicAdd(mine + (size_t)cur * A.ld, tot);
            tot = 0.f;
            cur = next;
        };
        xt::TileIt it;
        bool have = xt::tile_next(it, S.words, A.nwords, A.tile0);
        if (have) stage(it.J);
        for (int k = 0; have; ++k) {
            xt::TileIt nx = it;
            const bool more = xt::tile_next(nx, S.words, A.nwords, A.tile0);
            const bool fresh = more && nx.J != it.J;
            if (G::abuf == 2 && fresh) stage(nx.J);
            const int *tl = A.tile_lab + (size_t)it.g * kN;
            const int l0 = tl[0];
            const uint4 chg = A.tile_chg[it.g];
            if (l0 != cur) flush(l0);  // uniform: the columns are the same for every row
            if (!__all_sync(0xffffffffu, xt::wait(&S.acc_full, (uint32_t)(k & 1), abort))) {
                *abort = 1;
                break;
            }
            tc::fence_after();
            // the terms of 32 columns; where the class changes among them, one masked sum per class (a test per
            // column, unrolled, was 15 k clocks per tile: 128 branches of straight-line code)
            auto add = [&](uint32_t (&v)[32], unsigned w, int c0) {
#pragma unroll
                for (int q = 0; q < 32; ++q) v[q] = __float_as_uint(xt::ex2(__uint_as_float(v[q])));
                auto masked = [&](unsigned m) {
                    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
                    for (int q = 0; q < 32; q += 4) {
                        a0 += __uint_as_float(v[q] & (0u - (m >> q & 1u)));
                        a1 += __uint_as_float(v[q + 1] & (0u - (m >> (q + 1) & 1u)));
                        a2 += __uint_as_float(v[q + 2] & (0u - (m >> (q + 2) & 1u)));
                        a3 += __uint_as_float(v[q + 3] & (0u - (m >> (q + 3) & 1u)));
                    }
                    return (a0 + a1) + (a2 + a3);
                };
                if (w == 0u) {
                    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
                    for (int q = 0; q < 32; q += 4) {
                        a0 += __uint_as_float(v[q]);
                        a1 += __uint_as_float(v[q + 1]);
                        a2 += __uint_as_float(v[q + 2]);
                        a3 += __uint_as_float(v[q + 3]);
                    }
                    tot += (a0 + a1) + (a2 + a3);
                    return;
                }
                unsigned from = 0xffffffffu;  // columns of the current class and after
#pragma unroll 1
                while (w) {
                    const int q = __ffs(w) - 1;
                    w &= w - 1u;
                    const unsigned rest = 0xffffffffu << q;
                    tot += masked(from & ~rest);
                    flush(tl[c0 + q]);
                    from = rest;
                }
                tot += masked(from);
            };
            uint32_t va[32], vb[32];
            tc::ld32_async(lanes, va);
            tc::ld_wait(va);
            tc::ld32_async(lanes + 32, vb);
            add(va, chg.x, 0);
            tc::ld_wait(vb);
            tc::ld32_async(lanes + 64, va);
            add(vb, chg.y, 32);
            tc::ld_wait(va);
            tc::ld32_async(lanes + 96, vb);
            add(va, chg.z, 64);
            tc::ld_wait(vb);
            tc::fence_before();
            xt::arrive(&S.acc_free);
            add(vb, chg.w, 96);
            if (G::abuf == 1 && fresh) stage(nx.J);
            it = nx;
            have = more;
        }
        flush(A.L);
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (S.abort && t == 0) atomicOr(A.err, 1u);
    if (warp == 5) tc::tmem_dealloc(tmem, xt::kTmemCols);
}

// A row whose label is decided again: its place in the caller's order, its row of `score`, the tolerance of its scores.
struct Tie {
    int i, r;
    float tol;
};

// Row sums, argmax (lowest class on ties) and scores in the caller's order; rows outside the safe range are listed.
// f, cl: potential and cluster of a row; rad: radius of a cluster; umax: bits of the largest u.
__global__ void xfer_finish_kernel(const float *score, size_t ld, int n, int L, const int *perm, const float *f, const uint32_t *cl,
                                   const float *rad, const unsigned *umax, float s, float *sc_out, int *am_out, float *ms_out,
                                   int4 *fallback, int *n_fallback, Tie *ties, int *n_ties) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int i = perm[r];
    float tot = 0.f, best = -1.f, second = -1.f;
    int bestl = -1;
    for (int l = 0; l < L; ++l) {
        const float v = score[(size_t)l * ld + r];
        if (sc_out) sc_out[(size_t)i * L + l] = v;
        tot += v;
        if (v > best) {
            second = best;
            best = v;
            bestl = l;
        } else if (v > second) {
            second = v;
        }
    }
    if (!(tot >= 0x1p-60f && tot <= 0x1p60f)) {
        fallback[atomicAdd(n_fallback, 1)] = make_int4(r, 0, 0, 0);
        return;
    }
    am_out[i] = bestl;
    if (ms_out) ms_out[i] = tot;
    const float rc = rad[cl[r]], tol = fmaxf(kTie, kTieRel * s * (2.f * fabsf(f[r]) + __uint_as_float(*umax) + rc * rc));
    if (second > 0.f && best - second <= tol * best) ties[atomicAdd(n_ties, 1)] = Tie{i, r, tol};
}

__global__ void inverse_kernel(const int *perm, int n, int *inv) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) inv[perm[k]] = k;
}

// One CTA per listed row: the sums of the classes within the tolerance of the best one, as transport_gen_kernel forms them, then
// the argmax.  rows: packed in the caller's order (perm: the k-means order of that kernel); cols, logw, g: sorted by
// label, lab_off their classes.
struct TieArgs {
    const Tie *ties;
    const float *score;
    size_t ld;
    const float *rows, *f;
    const int *label, *perm, *inv, *off;
    const float *cols, *logw, *g;
    const int *lab_off;
    int D4, L;
    float eps, s;
    int *argmax;
};
__global__ void __launch_bounds__(256) xfer_tie_kernel(const __grid_constant__ TieArgs A) {
    __shared__ float cen[64], X[64], scores[1024], term[256];
    __shared__ int cand[1024], n_cand;
    __shared__ float m_s;
    const Tie tie = A.ties[blockIdx.x];
    const int t = threadIdx.x, D4 = A.D4, i = tie.i;
    if (t == 0) {  // the candidates in class order
        const float *sc = A.score + tie.r;
        float best = 0.f;
        int n = 0;
        for (int l = 0; l < A.L; ++l) best = fmaxf(best, sc[(size_t)l * A.ld]);
        for (int l = 0; l < A.L; ++l)
            if (best - sc[(size_t)l * A.ld] <= tie.tol * best) cand[n++] = l;
        n_cand = n;
    }
    const float s = A.s;
    const int c = A.label[i], a = A.off[c];
    const int r0 = a + (A.inv[i] - a) / 128 * 128, nr = min(A.off[c + 1] - r0, 128);
    if (t < D4) {
        float acc = 0.f;
        for (int r = 0; r < nr; ++r) acc += A.rows[(size_t)A.perm[r0 + r] * D4 + t];
        cen[t] = nr > 0 ? acc / (float)nr : 0.f;
        X[t] = A.rows[(size_t)i * D4 + t] - cen[t];
    }
    __syncthreads();
    if (t == 0) {
        float acc = 0.f;
        for (int k = 0; k < D4; ++k) acc = fmaf(X[k], X[k], acc);
        m_s = (float)((double)s * (0.5 * (double)acc - (double)A.f[i]));
    }
    __syncthreads();
    if (t < D4) X[t] *= s;
    __syncthreads();
    const float m = m_s;
    // terms of 256 columns at a time (one column per thread), then summed in that kernel's order: 16 threads, thread tc
    // adding (e0 + e1) + (e2 + e3) of columns 4 tc .. 4 tc + 3 of each 64
    for (int q = 0; q < n_cand; ++q) {
        const int lb = A.lab_off[cand[q]], le = A.lab_off[cand[q] + 1];
        float rs = 0.f;
        for (int p0 = lb; p0 < le; p0 += 256) {
            const int j = p0 + t;
            float h = -INFINITY;
            if (j < le) {
                const float4 *y4 = reinterpret_cast<const float4 *>(A.cols + (size_t)j * D4);
                float hn = 0.f;
#pragma unroll 4
                for (int k = 0; k < D4 / 4; ++k) {
                    const float4 v = y4[k];
                    const float y[4] = {v.x - cen[4 * k], v.y - cen[4 * k + 1], v.z - cen[4 * k + 2], v.w - cen[4 * k + 3]};
#pragma unroll
                    for (int u = 0; u < 4; ++u) hn = fmaf(y[u], y[u], hn);
                }
                h = __fsub_rn(__fmul_rn(s, fmaf(A.eps, A.logw[j], A.g[j]) - 0.5f * hn), m);  // two roundings
#pragma unroll 4
                for (int k = 0; k < D4 / 4; ++k) {
                    const float4 v = y4[k];
                    const float y[4] = {v.x - cen[4 * k], v.y - cen[4 * k + 1], v.z - cen[4 * k + 2], v.w - cen[4 * k + 3]};
#pragma unroll
                    for (int u = 0; u < 4; ++u) h = fmaf(X[4 * k + u], y[u], h);
                }
            }
            term[t] = xt::ex2(h);
            __syncthreads();
            if (t < 16)
                for (int u = 0; u < 256 && p0 + u < le; u += 64) {
                    const float *e = term + u + 4 * t;
                    rs += (e[0] + e[1]) + (e[2] + e[3]);
                }
            __syncthreads();
        }
        if (t < 32) {
            for (int o = 8; o > 0; o >>= 1) rs += __shfl_xor_sync(0xffffffffu, rs, o);
            if (t == 0) scores[q] = rs;
        }
    }
    __syncthreads();
    if (t == 0) {
        float best = -1.f;
        int bestl = -1;
        for (int q = 0; q < n_cand; ++q)
            if (scores[q] > best) {
                best = scores[q];
                bestl = cand[q];
            }
        A.argmax[i] = bestl;
    }
}

// The candidates of the listed rows (the classes within the tolerance of the best one) into their blocks' class bits, and the rows' marks.
// label: cluster of a row in the caller's order; blk0: first block of a cluster.
__global__ void xfer_mark_kernel(const Tie *ties, int n, const float *score, size_t ld, int L, const int *label, const int *off,
                                 const int *inv, const int *blk0, int words, unsigned *bits, unsigned char *tied) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const Tie tie = ties[k];
    const int i = tie.i, c = label[i], r = inv[i];
    const float *sc = score + tie.r;
    unsigned *b = bits + (size_t)(blk0[c] + (r - off[c]) / 128) * words;
    float best = 0.f;
    for (int l = 0; l < L; ++l) best = fmaxf(best, sc[(size_t)l * ld]);
    for (int l = 0; l < L; ++l)
        if (best - sc[(size_t)l * ld] <= tie.tol * best && !(b[l >> 5] >> (l & 31) & 1u)) atomicOr(b + (l >> 5), 1u << (l & 31));
    tied[r] = 1;
}

// sort keys of the columns: cluster, then label (L: ignored)
__global__ void xfer_keys_kernel(const int *cl, const int *labels, int m, int L, uint32_t *keys) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= m) return;
    const int l = labels[j];
    keys[j] = (uint32_t)cl[j] * (uint32_t)(L + 1) + (uint32_t)(l >= 0 && l < L ? l : L);
}
__global__ void xfer_labels_kernel(const uint32_t *keys, int m, int L, int *lab) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < m) lab[j] = (int)(keys[j] % (uint32_t)(L + 1));
}

template <int K> void sweep(const XferArgs &A, int nblk, cudaStream_t st) {
    constexpr int bytes = xt::Geom<3, K>::stages * xt::Geom<3, K>::tile + (int)sizeof(Ctl);
    static PerDevice<int> attr;
    attr.get([] {
        OTGB_CUDA_TRY(cudaFuncSetAttribute(xfer_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
        return 1;
    });
    xfer_tiles_kernel<K><<<A.ntiles, kN, 0, st>>>(A);
    OTGB_CHECK_LAUNCH();
    xfer_kernel<K><<<nblk, kThreads, bytes, st>>>(A);
    OTGB_CHECK_LAUNCH();
}

}  // namespace

TransportFallback transport_xt_apply(otgb_ctx *ctx, const TransportCall &c) {
    cudaStream_t st = ctx_stream(ctx);
    Workspace &ws = ctx_ws(ctx);
    const int N = c.N, M = c.M, D = c.D, L = c.L, D4 = (D + 3) & ~3;
    // Column clusters: about 512 columns (four tiles, so that the tail of a cluster's last tile is an eighth of its
    // work), but at least 32 of them, so that small atlases still tell their bundles apart.
    const int K = std::max(1, std::min(std::min(std::max(M / 512, 32), 2048), M));
    KmeansResult km = kmeans(ctx, "ta:km", c.y, nullptr, M, D, K, 2, 12345, nullptr, 16384);
    uint32_t *keys = ws.get<uint32_t>("ta:keys", M);
    int *cperm = ws.get<int>("ta:cperm", M);
    int *lab = ws.get<int>("ta:lab", M);
    void *scr = ws.get("sort:scratch", radix_sort_scratch_bytes(std::max(N, M)));
    xfer_keys_kernel<<<(M + 255) / 256, 256, 0, st>>>(km.labels, c.labels, M, L, keys);
    OTGB_CHECK_LAUNCH();
    int bits = 0;
    while ((1ll << bits) < (long long)K * (L + 1)) ++bits;
    radix_sort_pairs(keys, cperm, M, bits, scr, st);
    xfer_labels_kernel<<<(M + 255) / 256, 256, 0, st>>>(keys, M, L, lab);
    OTGB_CHECK_LAUNCH();
    // Row clusters of their own (the nearest column centroid is no compact set where a row bundle has no column bundle
    // near it: one such cluster visits every column, and its blocks are the launch's tail).
    const int Kr = std::max(1, std::min(std::min(std::max(N / 512, 32), 2048), N));
    KmeansResult ro = kmeans(ctx, "ta:kr", c.x, nullptr, N, D, Kr, 2, 12345, nullptr, 16384);
    std::vector<int> hc(K + 1), hr(Kr + 1);
    OTGB_CUDA_TRY(cudaMemcpyAsync(hc.data(), km.offsets, sizeof(int) * (K + 1), cudaMemcpyDeviceToHost, st));
    OTGB_CUDA_TRY(cudaMemcpyAsync(hr.data(), ro.offsets, sizeof(int) * (Kr + 1), cudaMemcpyDeviceToHost, st));

    float *C = ws.get<float>("ta:C", (size_t)M * D4), *Clw = ws.get<float>("ta:Clw", M), *Cw = ws.get<float>("ta:Cw", M);
    float *gs = ws.get<float>("ta:g", M), *R = ws.get<float>("ta:R", (size_t)N * D4), *Rw = ws.get<float>("ta:Rw", N);
    float *fs = ws.get<float>("ta:f", N);
    pack_points(c.y, c.b, cperm, M, D, c.d_cen, C, Clw, Cw, st);
    permute(c.g, cperm, M, gs, st);
    pack_points(c.x, nullptr, ro.perm, N, D, c.d_cen, R, nullptr, Rw, st);
    permute(c.f, ro.perm, N, fs, st);
    float *cen = ws.get<float>("ta:cen", (size_t)(K + Kr) * D4), *rad = ws.get<float>("ta:rad", K + Kr);
    float *mass = ws.get<float>("ta:mass", K + Kr), *mx = ws.get<float>("ta:max", K + Kr);
    float *rcen = cen + (size_t)K * D4, *rrad = rad + K;
    cluster_stats(C, D4, D, Cw, km.offsets, K, cen, D4, mass, rad, nullptr, st);
    cluster_stats(R, D4, D, Rw, ro.offsets, Kr, rcen, D4, mass + K, rrad, nullptr, st);
    const float eps = (float)c.eps, s = (float)(1.4426950408889634 / c.eps);
    int *nfb = ws.get<int>("ta:nfb", 3);  // fallback rows, near ties, bits of the largest u
    unsigned *umax = reinterpret_cast<unsigned *>(nfb + 2);
    OTGB_CUDA_TRY(cudaMemsetAsync(nfb, 0, 3 * sizeof(int), st));
    xfer_max_kernel<<<(K + 7) / 8, 256, 0, st>>>(km.offsets, K, gs, Clw, eps, mx, umax);
    OTGB_CHECK_LAUNCH();
    xfer_max_kernel<<<(Kr + 7) / 8, 256, 0, st>>>(ro.offsets, Kr, fs, nullptr, eps, mx + K, nullptr);
    OTGB_CHECK_LAUNCH();
    const int nwords = (K + 31) / 32;
    unsigned *kb = ws.get<unsigned>("ta:bits", (size_t)Kr * nwords);
    xfer_mask_kernel<<<Kr, 128, 0, st>>>(rcen, rrad, mx + K, cen, rad, mx, K, D4, s, kb, nwords);
    OTGB_CHECK_LAUNCH();

    // tiles of the column clusters and row blocks, from the offsets
    OTGB_CUDA_TRY(cudaStreamSynchronize(st));
    std::vector<int> up(K + 1), tcl, br, bc;
    up[0] = 0;
    for (int J = 0; J < K; ++J) {
        const int nt = (hc[J + 1] - hc[J] + kN - 1) / kN;
        tcl.insert(tcl.end(), nt, J);
        up[J + 1] = up[J] + nt;
    }
    for (int J = 0; J < Kr; ++J)
        for (int r = hr[J]; r < hr[J + 1]; r += xt::kRows) {
            br.push_back(r);
            bc.push_back(J);
        }
    br.push_back(N);
    const int ntiles = (int)tcl.size(), nblk = (int)bc.size();
    const size_t o_cl = up.size(), o_br = o_cl + tcl.size(), o_bc = o_br + br.size();
    up.insert(up.end(), tcl.begin(), tcl.end());
    up.insert(up.end(), br.begin(), br.end());
    up.insert(up.end(), bc.begin(), bc.end());
    int *d_up = ws.get<int>("ta:up", up.size());
    OTGB_CUDA_TRY(cudaMemcpyAsync(d_up, up.data(), sizeof(int) * up.size(), cudaMemcpyHostToDevice, st));

    XferArgs A;
    std::memset(&A, 0, sizeof(A));
    A.rows = R; A.f = fs; A.D4 = D4;
    A.blk_row0 = d_up + o_br; A.blk_cl = d_up + o_bc;
    A.bits = kb; A.nwords = nwords;
    A.tiles = static_cast<unsigned char *>(ws.get("ta:tiles", (size_t)ntiles * tcc_tile_bytes(3, D4)));
    float *hn = ws.get<float>("ta:hn", (size_t)ntiles * kN);
    A.half_norm = hn;
    A.tile0 = d_up; A.tile_cl = d_up + o_cl; A.off = km.offsets; A.ntiles = ntiles;
    A.ccen = cen; A.col_logw = Clw; A.g = gs; A.lab = lab;
    A.tile_lab = ws.get<int>("ta:tlab", (size_t)ntiles * kN);
    A.tile_chg = ws.get<uint4>("ta:tchg", ntiles);
    A.ld = ((size_t)N + 31) / 32 * 32;
    A.score = ws.get<float>("ta:sct", A.ld * L);
    A.L = L; A.eps = eps; A.s = s;
    A.err = ws.get<unsigned>("ta:err", 1);
    OTGB_CUDA_TRY(cudaMemsetAsync(A.score, 0, sizeof(float) * A.ld * L, st));
    OTGB_CUDA_TRY(cudaMemsetAsync(A.err, 0, sizeof(unsigned), st));
    tcc_build_side(3, C, D4, km.offsets, A.tile0, A.tile_cl, ntiles, cen, A.tiles, nullptr, hn, st);
    switch (xt::k_slots(D4)) {
        case 16: sweep<16>(A, nblk, st); break;
        case 32: sweep<32>(A, nblk, st); break;
        case 48: sweep<48>(A, nblk, st); break;
        case 64: sweep<64>(A, nblk, st); break;
        default: throw Error{OTGB_EINTERNAL, "transport_apply: unsupported width"};
    }
    int4 *fb = ws.get<int4>("ta:fb", N);
    Tie *ties = ws.get<Tie>("ta:ties", N);
    xfer_finish_kernel<<<(N + 127) / 128, 128, 0, st>>>(A.score, A.ld, N, L, ro.perm, fs, ro.sorted_keys, rrad, umax, s, c.scores,
                                                        c.argmax, c.row_mass, fb, nfb, ties, nfb + 1);
    OTGB_CHECK_LAUNCH();
    int *hp = static_cast<int *>(ctx_pinned(ctx));
    OTGB_CUDA_TRY(cudaMemcpyAsync(hp, nfb + 1, sizeof(int), cudaMemcpyDeviceToHost, st));
    OTGB_CUDA_TRY(cudaMemcpyAsync(hp + 1, A.err, sizeof(unsigned), cudaMemcpyDeviceToHost, st));
    OTGB_CUDA_TRY(cudaStreamSynchronize(st));
    require(hp[1] == 0, "transport_apply: a bounded device wait gave up", OTGB_ETIMEOUT);
    const int n_ties = hp[0];
    const TransportFallback out{R, fs, C, Clw, gs, lab, ro.perm, fb, nfb};
    if (n_ties <= 0) return out;

    // the orders of the CUDA-core kernel: columns by label, rows by a k-means of N / 64 clusters
    const int Kt = std::max(1, std::min(N / 64, 4096));
    KmeansResult kt = kmeans(ctx, "ta:kt", c.x, nullptr, N, D, Kt, 4, 12345, nullptr);
    uint32_t *k2 = ws.get<uint32_t>("ta:keys2", M);
    int *perm2 = ws.get<int>("ta:cperm2", M), *lab_off = ws.get<int>("ta:laboff", L + 1), *inv = ws.get<int>("ta:inv", N);
    float *C2 = ws.get<float>("ta:C2", (size_t)M * D4), *lw2 = ws.get<float>("ta:Clw2", M), *g2 = ws.get<float>("ta:g2", M);
    float *R2 = ws.get<float>("ta:R2", (size_t)N * D4);
    label_order(ctx, c.labels, M, L, k2, perm2, lab_off);
    pack_points(c.y, c.b, perm2, M, D, c.d_cen, C2, lw2, nullptr, st);
    permute(c.g, perm2, M, g2, st);
    inverse_kernel<<<(N + 255) / 256, 256, 0, st>>>(kt.perm, N, inv);
    OTGB_CHECK_LAUNCH();
    if (n_ties <= kFewTies) {  // a CTA per row
        pack_points(c.x, nullptr, nullptr, N, D, c.d_cen, R2, nullptr, nullptr, st);
        const TieArgs T{ties, A.score, A.ld, R2, c.f, kt.labels, kt.perm, inv, kt.offsets, C2, lw2, g2, lab_off, D4, L, eps, s, c.argmax};
        xfer_tie_kernel<<<n_ties, 256, 0, st>>>(T);
        OTGB_CHECK_LAUNCH();
        return out;
    }
    // the kernel itself, over the blocks and classes that are concerned
    std::vector<int> off(Kt + 1), b0(Kt), rows;
    OTGB_CUDA_TRY(cudaMemcpyAsync(off.data(), kt.offsets, sizeof(int) * (Kt + 1), cudaMemcpyDeviceToHost, st));
    pack_points(c.x, nullptr, kt.perm, N, D, c.d_cen, R2, nullptr, nullptr, st);
    float *f2 = ws.get<float>("ta:f2", N);
    permute(c.f, kt.perm, N, f2, st);
    OTGB_CUDA_TRY(cudaStreamSynchronize(st));
    for (int q = 0; q < Kt; ++q) {
        b0[q] = (int)rows.size();
        for (int r = off[q]; r < off[q + 1]; r += 128) rows.push_back(r);
    }
    const int nb = (int)rows.size(), words = (L + 31) / 32;
    rows.push_back(N);
    rows.insert(rows.end(), b0.begin(), b0.end());
    int *d_rows = ws.get<int>("ta:blk2", rows.size());
    unsigned *bits2 = ws.get<unsigned>("ta:cls", (size_t)nb * words);
    unsigned char *tied = ws.get<unsigned char>("ta:tied", N);
    OTGB_CUDA_TRY(cudaMemcpyAsync(d_rows, rows.data(), sizeof(int) * rows.size(), cudaMemcpyHostToDevice, st));
    OTGB_CUDA_TRY(cudaMemsetAsync(bits2, 0, sizeof(unsigned) * nb * words, st));
    OTGB_CUDA_TRY(cudaMemsetAsync(tied, 0, N, st));
    xfer_mark_kernel<<<(n_ties + 255) / 256, 256, 0, st>>>(ties, n_ties, A.score, A.ld, L, kt.labels, kt.offsets, inv,
                                                          d_rows + nb + 1, words, bits2, tied);
    OTGB_CHECK_LAUNCH();
    transport_gen_ties(TieBlocks{R2, f2, C2, lw2, g2, d_rows, lab_off, kt.perm, nb, N, M, D, L, eps, s, bits2, tied, c.argmax}, st);
    OTGB_CUDA_TRY(cudaStreamSynchronize(st));  // the host vector goes out of scope
    return out;
}

}  // namespace otgb
