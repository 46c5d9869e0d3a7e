// Large dense D <= 3 sums over spatially sorted points: otgb_softmin (tensor cores) and the gradient in the points (packed
// float32).
//
// Rows and columns come in the order of a Hilbert curve, so that a block of 128 rows and a tile of 128 columns are compact.
// A CTA bounds the exponents of every tile from the boxes of the block and the tile and the tile's largest
// s (eps log w + pot), visits the best tile first, and then only the tiles whose bound reaches to 60 binades below the
// smallest running shift of its rows: a term below 2^-60 of the row's largest one changes neither a float32 sum of fewer than
// 2^31 terms nor a weighted mean of it (the exponents in between are visited, whatever the potentials are, so nothing depends
// on their being near a solution).  On voxels at blur 1 that leaves about one pair in eight.
//
// softmin3_sorted_kernel: the exponent of a pair is one K = 32 tensor-core dot product (tile3.cuh); one thread per row keeps
// a running shift and the sum.  The curve jumps where the points leave gaps, so a block is cut into runs whose box stays
// compact (s times its squared half diagonal at most kCompact): groups of 16 rows, each cut once more at its longest step, are
// merged in order while their box allows it.  The runs take their turns on the CTA, each with its own centre and its own
// tiles: a block across a jump costs two short passes instead of one that visits everything between.  A single part above
// kSpread (outliers: the dot product's terms would dwarf the exponents) is summed from coordinate differences alone.  Where
// that comes to more passes than one over all tiles (points so sparse at the blur, or so far from each other's cells of the
// curve, that every part is loose) both limits grow by eights until it does not or a few passes are left, as far as one run
// for the block, which is what the dense sweep has: 100k points on a line, eps 0.01, 21 -> 0.9 ms (CUDA cores 7.0); 100k points with one outlier that
// takes the curve's resolution 135 -> 4.2 (7.3).
// Bound: MUFU, 32 pairs per clock and SM.  otgb_softmin on 100k x 100k voxels 0.83 ms, of it 0.55 the sums (ex2 at 51 % of the
// MUFU, issue 66 % of the active clocks); the dense tensor-core sweep 1.87, the CUDA cores 7.0.
//
// grad3_sorted_kernel: the whole block in one run, in coordinate differences (two columns per packed f32x2 operation, a
// running shift per row, the tile's coordinates read as broadcasts).  The gradient is a small difference of two large sums:
// on the tensor cores it needed runs with s (half diagonal)^2 below 12 to stay near the CUDA cores' error (1.0e-6; 1.1e-6),
// up to sixteen passes a block, and was slower than grad_kernel where blocks are loose (2,000 + 2,000 points 0.53 against
// 0.35 ms, 20,000 + 20,000 with one far outlier, which takes the curve's whole resolution, 14 against 3.4).  Differences
// need no compact runs, and a block that is loose only visits more tiles.
// Bound: the FP32 pipe, 11 operations per pair (3 differences, 4 for the exponent, 1 shift, 3 sums; ex2 takes 4 of its
// clocks): 3.7e12 pairs/s.  Every pair of 50k + 50k points (far outlier) 76 -> 2.5 ms = 2.0e12; the FP32 pipe and
// fixed-latency waits are the largest stalls.  sinkhorn_grad_x on 50k + 50k voxels 2.17 -> 1.24 ms, of it 1.01 the sums
// (grad_kernel 8.6), error 9.7e-7 -> 4.6e-7; 2,000 + 2,000 points 0.53 -> 0.17.
//
// Each (block, split, part) writes its shift and sums; a finish kernel combines the splits in order, so the result does
// not depend on scheduling.
#include <cfloat>
#include <cmath>
#include <cstring>

#include "prims.cuh"
#include "solver.cuh"
#include "sorted3.cuh"
#include "tile3.cuh"

namespace otgb {
namespace {

constexpr int kT = 128;           // threads, rows of a block, columns of a tile
constexpr int kMaxTiles = 4096;   // tiles bounded at once (524,288 columns)
constexpr float kNoTerm = -1e29f;
constexpr float kReach = 60.f;    // binades below the row's largest term that are visited
// s (half diagonal)^2 of a run: what the products of the exponent are rounded at (error 7e-8 at 96)
constexpr float kCompact = 96.f;
constexpr int kPasses = 12;       // of a block's runs (one outside kSpread counts four): above, they are made larger,
constexpr int kFewPasses = 6;     // and where together they visit more than every tile once: up to this number by one step only
constexpr float kSpread = 256.f;  // terms of this size are rounded at 8e-6, as s f + s g - s C is at |s f| = 128

struct S3Part {
    const float4 *cols;
    const float *pot;
    const float4 *box;  // per tile: (lo, largest s (eps log w + pot)), (hi, 0)
    int n;
};
struct S3Args {
    const float4 *rows;
    int n_rows, splits;
    S3Part part[2];
    float eps, s;
    float4 *out;  // [part][split][row]: shift, then S (softmin) or the three sums
    unsigned *err;  // softmin
};

// Bounds and visit list of one window of tiles.
struct Visit {
    float bnd[kMaxTiles];
    unsigned short list[kMaxTiles];
    float best[4];
    int ibest[4], wsum[4];
};
struct S3Smem {
    unsigned char a[t3::kBytes], b[t3::kBytes];
    alignas(16) float ys[3][kT];
    float ct[kT];  // s (eps log w + pot), for a spread block
    Visit v;
    float red[4];
    float sub[16][6];  // boxes of the two parts of each group of 16 rows: lo, -hi
    int start[17];     // their first rows
    unsigned long long mbar;
    uint32_t tslot;
};

// Bounds of tiles w0 .. w0 + nw - 1 for rows within [lo, hi]; returns the best tile, relative to w0.  CTA-collective.
__device__ __forceinline__ int bound_tiles(Visit &V, const float4 *box, int w0, int nw, const float (&lo)[3], const float (&hi)[3],
                                           float s) {
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    float best = -INFINITY;
    int bi = 0x7fffffff;
    for (int q = t; q < nw; q += kT) {
        const float4 l = box[2 * (w0 + q)], h = box[2 * (w0 + q) + 1];
        const float g0 = fmaxf(fmaxf(l.x - hi[0], lo[0] - h.x), 0.f), g1 = fmaxf(fmaxf(l.y - hi[1], lo[1] - h.y), 0.f),
                    g2 = fmaxf(fmaxf(l.z - hi[2], lo[2] - h.z), 0.f);
        const float b = l.w - 0.49999f * s * fmaf(g0, g0, fmaf(g1, g1, g2 * g2));
        V.bnd[q] = b;
        if (b > best) {
            best = b;
            bi = q;
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi < bi)) {
            best = ob;
            bi = oi;
        }
    }
    if (lane == 0) {
        V.best[warp] = best;
        V.ibest[warp] = bi;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (q == 0) {
            best = V.best[0];
            bi = V.ibest[0];
        } else if (V.best[q] > best || (V.best[q] == best && V.ibest[q] < bi)) {
            best = V.best[q];
            bi = V.ibest[q];
        }
    }
    return bi == 0x7fffffff ? 0 : bi;  // 0: every bound is -inf or NaN
}

// Lists the tiles of [qa, qb) other than `skip` whose bound reaches thr (a NaN bound does), in order; returns their number.
// CTA-collective.
__device__ __forceinline__ int list_tiles(Visit &V, int qa, int qb, int skip, float thr) {
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int len = max(qb - qa, 0), each = (len + kT - 1) / kT, i0 = min(qa + t * each, qb), i1 = min(i0 + each, qb);
    int cnt = 0;
    for (int q = i0; q < i1; ++q) cnt += q != skip && !(V.bnd[q] < thr);
    int inc = cnt;
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) V.wsum[warp] = inc;
    __syncthreads();
    int pos = inc - cnt;
    for (int q = 0; q < warp; ++q) pos += V.wsum[q];
    const int n = V.wsum[0] + V.wsum[1] + V.wsum[2] + V.wsum[3];
    for (int q = i0; q < i1; ++q)
        if (q != skip && !(V.bnd[q] < thr)) V.list[pos++] = (unsigned short)q;
    __syncthreads();
    return n;
}
// The first list entry from k on that still reaches the shift.
__device__ __forceinline__ int next_tile(const Visit &V, int k, int n, float thr) {
    while (k < n && V.bnd[V.list[k]] < thr) ++k;
    return k;
}

__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ float sum2(unsigned long long v) {
    float lo, hi;
    unpack2(v, lo, hi);
    return lo + hi;
}

__global__ void __launch_bounds__(kT, 4) softmin3_sorted_kernel(const __grid_constant__ S3Args A) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    S3Smem &M = *reinterpret_cast<S3Smem *>(smem_raw);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int r0 = blockIdx.x * kT, nr = min(kT, A.n_rows - r0);
    const S3Part &P = A.part[0];
    const float s = A.s;
    const bool valid = t < nr;
    const int ntiles = (P.n + kT - 1) / kT;

    // ---- the groups of 16 rows, cut at their longest step, and the boxes of the parts
    const float4 mine = A.rows[r0 + (valid ? t : 0)];
    {
        const int u = t & 15;
        const float px = __shfl_up_sync(0xffffffffu, mine.x, 1), py = __shfl_up_sync(0xffffffffu, mine.y, 1),
                    pz = __shfl_up_sync(0xffffffffu, mine.z, 1);
        const float e0 = mine.x - px, e1 = mine.y - py, e2 = mine.z - pz;
        float len = fmaf(e0, e0, fmaf(e1, e1, e2 * e2));
        if (!(len >= 0.f)) len = INFINITY;  // a row that is no number: all lanes agree on the cut
        if (u == 0 || !valid) len = -1.f;
        int cut = u;
        for (int o = 8; o > 0; o >>= 1) {
            const float ol = __shfl_xor_sync(0xffffffffu, len, o);
            const int oc = __shfl_xor_sync(0xffffffffu, cut, o);
            if (ol > len || (ol == len && oc < cut)) {
                len = ol;
                cut = oc;
            }
        }
        if (len < 0.f) cut = 16;  // a group of at most one row
        const int g = t >> 4;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const bool in = valid && (h ? u >= cut : u < cut);
            float v[6] = {mine.x, mine.y, mine.z, -mine.x, -mine.y, -mine.z};
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                v[q] = in ? v[q] : FLT_MAX;
                for (int o = 8; o > 0; o >>= 1) v[q] = fminf(v[q], __shfl_xor_sync(0xffffffffu, v[q], o));
                if (u == 0) M.sub[2 * g + h][q] = v[q];
            }
            if (u == 0) M.start[2 * g + h] = min(nr, 16 * g + (h ? cut : 0));
        }
        if (t == 0) M.start[16] = nr;
    }
    if (t == 0) {
        tc::mbar_init(&M.mbar, 1);
        tc::mbar_init_fence();
    }
    if (warp == 0) tc::tmem_alloc(&M.tslot, kT);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = M.tslot, lanes = tmem + ((uint32_t)(warp * 32) << 16);
    bool ok = true;
    int phase = 0;
    float4 rq = make_float4(0.f, 0.f, 0.f, 0.f);
    float rpot = 0.f;
    bool rin = false;
    float limit = kCompact;
    // The run that starts at part ga: its box; the part after it.
    auto extent = [&](int ga, float (&lo)[3], float (&hi)[3], bool &spread) -> int {
        float hd2 = 0.f;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            lo[d] = M.sub[ga][d];
            hi[d] = -M.sub[ga][d + 3];
            hd2 = fmaf(0.25f * (hi[d] - lo[d]), hi[d] - lo[d], hd2);
        }
        spread = !(s * hd2 <= limit * (kSpread / kCompact));
        int gb = ga + 1;
        for (; gb < 16 && !spread; ++gb) {
            if (M.start[gb] >= M.start[gb + 1]) continue;
            float l[3], h[3], u = 0.f;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                l[d] = fminf(lo[d], M.sub[gb][d]);
                h[d] = fmaxf(hi[d], -M.sub[gb][d + 3]);
                u = fmaf(0.25f * (h[d] - l[d]), h[d] - l[d], u);
            }
            if (!(s * u <= limit)) break;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                lo[d] = l[d];
                hi[d] = h[d];
            }
        }
        return gb;
    };
    // What the runs cost, in passes over the tiles.  Where that is too much the limit grows: larger runs, fewer passes; a block
    // across a jump of the curve stays cut there as long as any other one.
    auto count = [&]() -> int {
        int n = 0;
        bool finite = true;
        for (int ga = 0; ga < 16;) {
            if (M.start[ga] >= M.start[ga + 1]) {
                ++ga;
                continue;
            }
            float lo[3], hi[3];
            bool spread;
            ga = extent(ga, lo, hi, spread);
            n += spread ? 4 : 1;
            for (int d = 0; d < 3; ++d) finite = finite && hi[d] - lo[d] <= FLT_MAX;
        }
        return finite ? n : 1;  // no larger runs around a part without a centre
    };
    int passes = count();
    while (passes > kPasses && limit < 1e30f) {
        limit *= 8.f;
        passes = count();
    }
    for (int ga = 0, gb; ok && ga < 16; ga = gb) {
    // ---- the run of parts [ga, gb): box, centre, row operand
    if (M.start[ga] >= M.start[ga + 1]) {  // an empty part (uniform)
        gb = ga + 1;
        continue;
    }
    float lo[3], hi[3];
    bool spread;  // uniform
    gb = extent(ga, lo, hi, spread);
    const int ra = M.start[ga], rb = M.start[gb];
    const bool in_run = t >= ra && t < rb;
    const bool warp_on = 32 * warp < rb && 32 * warp + 32 > ra;  // some of the warp's rows are in the run
    const float4 p = in_run ? mine : A.rows[r0 + ra];  // the other threads repeat the run's first row
    const float c[3] = {0.5f * (lo[0] + hi[0]), 0.5f * (lo[1] + hi[1]), 0.5f * (lo[2] + hi[2])};
    {
        uint32_t w[16];
        t3::row_words(p.x - c[0], p.y - c[1], p.z - c[2], s, w);
        t3::store_words(M.a, t, w);
    }
    // S2: sum of one tile; S with what its additions lost (Kahan): of the tiles before.  A single chain over all columns drops
    // terms that are small beside the sum so far: 46,000 x 47,000 points of a square were off by 3.4e-6 (rms, blur 0.05; CUDA
    // cores 1.4e-6), now 6.4e-7.
    float sh = kNoTerm, S = 0.f, Slost = 0.f;
    unsigned long long S2 = 0ull;
    auto rescale = [&](float m) {
        const float f = xt::ex2(sh - m);
        S2 = mul2(S2, pack2(f, f));
        S *= f;
        Slost *= f;
        sh = m;
    };
    auto end_tile = [&] {
        const float u = sum2(S2) - Slost, z = S + u;
        Slost = (z - S) - u;
        S = z;
        S2 = 0ull;
    };
    auto load_raw = [&](int tile) {
        const int j = tile * kT + t;
        rin = tile >= 0 && j < P.n;
        if (rin) {
            rq = P.cols[j];
            rpot = P.pot[j];
        }
    };
    auto chunk = [&](const uint32_t (&v)[32]) {
        float m0 = __uint_as_float(v[0]), m1 = __uint_as_float(v[1]);
#pragma unroll
        for (int q = 2; q < 32; q += 2) {
            m0 = fmaxf(m0, __uint_as_float(v[q]));
            m1 = fmaxf(m1, __uint_as_float(v[q + 1]));
        }
        m0 = fmaxf(m0, m1);
        if (m0 > sh + 30.f) rescale(m0);
#pragma unroll
        for (int q = 0; q < 32; q += 2)
            S2 = add2(S2, pack2(xt::ex2(__uint_as_float(v[q]) - sh), xt::ex2(__uint_as_float(v[q + 1]) - sh)));
    };
    // one tile from registers: operand, MMA, sums; `next` is fetched meanwhile (-1: none).  Returns the smallest shift of
    // the block's rows.
    auto tile_step = [&](int next) -> float {
        if (spread) {
            M.ys[0][t] = -rq.x;
            M.ys[1][t] = -rq.y;
            M.ys[2][t] = -rq.z;
            M.ct[t] = rin ? s * fmaf(A.eps, rq.w, rpot) : -INFINITY;
            load_raw(next);
            __syncthreads();
            for (int q = 0; warp_on && q < kT; ++q) {
                const float ct = M.ct[q];
                if (ct == -INFINITY) continue;  // uniform
                const float d0 = p.x + M.ys[0][q], d1 = p.y + M.ys[1][q], d2 = p.z + M.ys[2][q];
                const float e = fmaf(-0.5f * s, fmaf(d0, d0, fmaf(d1, d1, d2 * d2)), ct);
                if (e > sh + 30.f) rescale(e);
                S2 = add2(S2, pack2(xt::ex2(e - sh), 0.f));
            }
            end_tile();
            float m = warp_on ? sh : INFINITY;
            for (int o = 16; o > 0; o >>= 1) m = fminf(m, __shfl_xor_sync(0xffffffffu, m, o));
            if (lane == 0) M.red[warp] = m;
            __syncthreads();
            return fminf(fminf(M.red[0], M.red[1]), fminf(M.red[2], M.red[3]));
        }
        const float y0 = rin ? rq.x - c[0] : 0.f, y1 = rin ? rq.y - c[1] : 0.f, y2 = rin ? rq.z - c[2] : 0.f;
        {
            uint32_t w[16];
            t3::col_words(y0, y1, y2, rq.w, rpot, s, A.eps, rin, w);
            t3::store_words(M.b, t, w);
        }
        load_raw(next);
        tc::fence_proxy_async();
        tc::fence_before();
        __syncthreads();
        tc::fence_after();
        if (t == 0) t3::issue(tmem, tc::smem_u32(M.a), tc::smem_u32(M.b), &M.mbar);
        if (!tc::mbar_wait(&M.mbar, (uint32_t)(phase & 1))) ok = false;
        ++phase;
        ok = __all_sync(0xffffffffu, ok);  // tensor-memory loads are warp-collective
        tc::fence_after();
        if (ok && warp_on) {
            uint32_t va[32], vb[32];
            tc::ld32_async(lanes, va);
            tc::ld_wait(va);
            tc::ld32_async(lanes + 32, vb);
            chunk(va);
            tc::ld_wait(vb);
            tc::ld32_async(lanes + 64, va);
            chunk(vb);
            tc::ld_wait(va);
            tc::ld32_async(lanes + 96, vb);
            chunk(va);
            tc::ld_wait(vb);
            chunk(vb);
        }
        end_tile();
        float m = warp_on ? sh : INFINITY;  // threads outside the run repeat one of its rows
        for (int o = 16; o > 0; o >>= 1) m = fminf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) M.red[warp] = m;
        tc::fence_before();
        ok = __syncthreads_and(ok) != 0;  // operand, coordinates and accumulator are free again
        return fminf(fminf(M.red[0], M.red[1]), fminf(M.red[2], M.red[3]));
    };

    // the tiles of this split (all of them are bounded, so that every split starts from the same best tile)
    const int per = (ntiles + A.splits - 1) / A.splits, ta = blockIdx.y * per, tb = min(ntiles, ta + per);
    float thr = -INFINITY;
    bool restart = false;
    for (int w0 = 0; ok && w0 < ntiles; w0 += kMaxTiles) {
        if (w0 > 0 && (w0 >= tb || w0 + kMaxTiles <= ta)) continue;  // none of this split's tiles
        const int nw = min(kMaxTiles, ntiles - w0);
        const int bi = bound_tiles(M.v, P.box, w0, nw, lo, hi, s);
        const bool own = w0 + bi >= ta && w0 + bi < tb;
        if (own || w0 == 0) {
            load_raw(w0 + bi);
            thr = tile_step(-1) - kReach;
            if (!ok) break;
            if (!own) {  // another split's tile: it only set the shift
                S = Slost = 0.f;
            }
        }
        // the other tiles of this split that can matter, in order (a NaN bound is visited)
        const int n_list = list_tiles(M.v, max(ta - w0, 0), min(tb - w0, nw), bi, thr);
        if (passes > 1 && passes * n_list > tb - ta && limit < (passes > kFewPasses ? 1e30f : kCompact * 8.f)) {
            restart = true;
            break;
        }
        int k = next_tile(M.v, 0, n_list, thr);
        if (k < n_list) load_raw(w0 + M.v.list[k]);
        while (ok && k < n_list) {
            const int nx = next_tile(M.v, k + 1, n_list, thr);
            thr = tile_step(nx < n_list ? w0 + M.v.list[nx] : -1) - kReach;
            k = nx;
        }
        __syncthreads();  // the next window overwrites the bounds
    }
    if (restart) {  // from the first part, in fewer runs
        for (const int before = passes; passes == before && limit < (before > kFewPasses ? 1e30f : kCompact * 8.f);) {
            limit *= 8.f;
            passes = count();
        }
        gb = 0;
        continue;
    }
    if (in_run) {
        const float x0 = p.x - c[0], x1 = p.y - c[1], x2 = p.z - c[2];
        const bool far_row = !spread && s * fmaf(x0, x0, fmaf(x1, x1, x2 * x2)) > xt::kFarRow;  // NaN: the safe kernel's row
        A.out[(size_t)blockIdx.y * A.n_rows + r0 + t] = make_float4(sh, far_row ? NAN : S - Slost, 0.f, 0.f);
    }
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (!ok && t == 0) atomicOr(A.err, 1u);
    if (warp == 0) tc::tmem_dealloc(tmem, kT);
}

// One CTA per block of 128 rows, split and part: the rows of the block as one run, in coordinate differences.
struct G3Smem {
    alignas(16) float y[2][4][kT];  // two tiles: -y per coordinate, s (eps log w + pot)
    Visit v;
    float red[2][4], box[4][6];
};

__global__ void __launch_bounds__(kT, 5) grad3_sorted_kernel(const __grid_constant__ S3Args A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    G3Smem &M = *reinterpret_cast<G3Smem *>(smem_raw);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int r0 = blockIdx.x * kT, nr = min(kT, A.n_rows - r0);
    const S3Part &P = A.part[blockIdx.z];
    const float s = A.s;
    const int ntiles = (P.n + kT - 1) / kT;
    const float4 p = A.rows[r0 + (t < nr ? t : 0)];  // threads without a row repeat the first one
    {
        float v[6] = {p.x, p.y, p.z, -p.x, -p.y, -p.z};
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            for (int o = 16; o > 0; o >>= 1) v[q] = fminf(v[q], __shfl_xor_sync(0xffffffffu, v[q], o));
            if (lane == 0) M.box[warp][q] = v[q];
        }
    }
    __syncthreads();
    float lo[3], hi[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        lo[d] = fminf(fminf(M.box[0][d], M.box[1][d]), fminf(M.box[2][d], M.box[3][d]));
        hi[d] = -fminf(fminf(M.box[0][d + 3], M.box[1][d + 3]), fminf(M.box[2][d + 3], M.box[3][d + 3]));
    }
    const unsigned long long X2[3] = {pack2(p.x, p.x), pack2(p.y, p.y), pack2(p.z, p.z)};
    const unsigned long long H2 = pack2(-0.5f * s, -0.5f * s);
    float sh = kNoTerm, W[3] = {0.f, 0.f, 0.f};
    float4 rq = make_float4(0.f, 0.f, 0.f, 0.f);
    float rpot = 0.f;
    bool rin = false;
    auto load_raw = [&](int tile) {
        const int j = tile * kT + t;
        rin = tile >= 0 && j < P.n;
        if (rin) {
            rq = P.cols[j];
            rpot = P.pot[j];
        }
    };
    int buf = 0;  // the tile in registers goes into this buffer
    auto store = [&] {
        const float ct = rin ? s * fmaf(A.eps, rq.w, rpot) : -INFINITY;
        const bool some = !(ct == -INFINITY);  // an absent column, or one without weight: its term is 0 whatever it holds
        M.y[buf][0][t] = some ? -rq.x : 0.f;
        M.y[buf][1][t] = some ? -rq.y : 0.f;
        M.y[buf][2][t] = some ? -rq.z : 0.f;
        M.y[buf][3][t] = ct;
    };
    // The sums of the tile in buffer b, added to W; the smallest shift of the warp into red[b].
    auto sums = [&](int b) {
        unsigned long long V[3] = {0ull, 0ull, 0ull};
        const float(*y)[kT] = M.y[b];
#pragma unroll 1
        for (int q = 0; q < kT; q += 8) {
            unsigned long long D[3][4], E[4];
#pragma unroll
            for (int d = 0; d < 3; ++d)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const ulonglong2 u = *reinterpret_cast<const ulonglong2 *>(&y[d][q + 4 * h]);
                    D[d][2 * h] = add2(X2[d], u.x);
                    D[d][2 * h + 1] = add2(X2[d], u.y);
                }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const ulonglong2 u = *reinterpret_cast<const ulonglong2 *>(&y[3][q + 4 * h]);
                E[2 * h] = u.x;
                E[2 * h + 1] = u.y;
            }
            float e[8];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                E[h] = fma2(H2, fma2(D[2][h], D[2][h], fma2(D[1][h], D[1][h], mul2(D[0][h], D[0][h]))), E[h]);
                unpack2(E[h], e[2 * h], e[2 * h + 1]);
            }
            const float m = fmaxf(fmaxf(fmaxf(e[0], e[1]), fmaxf(e[2], e[3])), fmaxf(fmaxf(e[4], e[5]), fmaxf(e[6], e[7])));
            if (m > sh + 30.f) {
                const float f = xt::ex2(sh - m);
                const unsigned long long ff = pack2(f, f);
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    V[d] = mul2(V[d], ff);
                    W[d] *= f;
                }
                sh = m;
            }
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const unsigned long long w = pack2(xt::ex2(e[2 * h] - sh), xt::ex2(e[2 * h + 1] - sh));
#pragma unroll
                for (int d = 0; d < 3; ++d) V[d] = fma2(w, D[d][h], V[d]);
            }
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) W[d] += sum2(V[d]);
        float m = sh;
        for (int o = 16; o > 0; o >>= 1) m = fminf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) M.red[b][warp] = m;
    };
    auto reached = [&](int b) { return fminf(fminf(M.red[b][0], M.red[b][1]), fminf(M.red[b][2], M.red[b][3])) - kReach; };

    const int per = (ntiles + A.splits - 1) / A.splits, ta = blockIdx.y * per, tb = min(ntiles, ta + per);
    float thr = -INFINITY;
    for (int w0 = 0; w0 < ntiles; w0 += kMaxTiles) {
        if (w0 > 0 && (w0 >= tb || w0 + kMaxTiles <= ta)) continue;  // none of this split's tiles
        const int nw = min(kMaxTiles, ntiles - w0);
        const int bi = bound_tiles(M.v, P.box, w0, nw, lo, hi, s);
        const bool own = w0 + bi >= ta && w0 + bi < tb;
        if (own || w0 == 0) {
            load_raw(w0 + bi);
            store();
            __syncthreads();
            sums(buf);
            __syncthreads();
            thr = reached(buf);
            buf ^= 1;
            if (!own) W[0] = W[1] = W[2] = 0.f;  // another split's tile: it only set the shift
        }
        const int n_list = list_tiles(M.v, max(ta - w0, 0), min(tb - w0, nw), bi, thr);
        int k = next_tile(M.v, 0, n_list, thr);
        if (k < n_list) load_raw(w0 + M.v.list[k]);
        bool first = true;
        while (k < n_list) {
            store();
            // one barrier per tile: every thread is past the sums of the tile before (the other buffer), whose shift the choice
            // of the next tile may use; this buffer was last read before the barrier before
            __syncthreads();
            if (!first) thr = fmaxf(thr, reached(buf ^ 1));
            first = false;
            const int nx = next_tile(M.v, k + 1, n_list, thr);
            load_raw(nx < n_list ? w0 + M.v.list[nx] : -1);
            sums(buf);
            buf ^= 1;
            k = nx;
        }
        __syncthreads();  // the next window overwrites the bounds
    }
    if (t < nr) A.out[((size_t)blockIdx.z * A.splits + blockIdx.y) * A.n_rows + r0 + t] = make_float4(sh, W[0], W[1], W[2]);
}

// Boxes of the column tiles of both parts (blockIdx.y), one warp per tile.
__global__ void tile_box_kernel(const __grid_constant__ S3Args A, float4 *box0, float4 *box1) {
    const S3Part &P = A.part[blockIdx.y];
    float4 *box = blockIdx.y ? box1 : box0;
    const int g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (g * kT >= P.n) return;
    float v[6] = {FLT_MAX, FLT_MAX, FLT_MAX, FLT_MAX, FLT_MAX, FLT_MAX}, m = -INFINITY;
    for (int j = g * kT + lane; j < min(P.n, g * kT + kT); j += 32) {
        const float4 q = P.cols[j];
        v[0] = fminf(v[0], q.x); v[1] = fminf(v[1], q.y); v[2] = fminf(v[2], q.z);
        v[3] = fminf(v[3], -q.x); v[4] = fminf(v[4], -q.y); v[5] = fminf(v[5], -q.z);
        const float u = A.s * fmaf(A.eps, q.w, P.pot[j]);
        const bool num = u == u && q.x == q.x && q.y == q.y && q.z == q.z;
        m = num ? fmaxf(m, u) : INFINITY;  // a column that is not a number is visited by every row
    }
#pragma unroll
    for (int q = 0; q < 6; ++q)
        for (int o = 16; o > 0; o >>= 1) v[q] = fminf(v[q], __shfl_xor_sync(0xffffffffu, v[q], o));
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) {
        box[2 * g] = make_float4(v[0], v[1], v[2], m);
        box[2 * g + 1] = make_float4(-v[3], -v[4], -v[5], 0.f);
    }
}

struct GradFinish {
    const float4 *part;
    int n, D, splits;
    const float *row_pot[2];
    float sign[2];
    const float *row_w;
    const int *perm;
    float s, scale;
    int accumulate;
    float *grad;
};
__global__ void grad3_finish_kernel(const __grid_constant__ GradFinish F) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= F.n) return;
    float out[3] = {0.f, 0.f, 0.f};
    for (int q = 0; q < 2; ++q) {
        const float4 *p = F.part + (size_t)q * F.splits * F.n + r;
        float m = kNoTerm;
        for (int k = 0; k < F.splits; ++k) m = fmaxf(m, p[(size_t)k * F.n].x);
        if (!(m > kNoTerm)) continue;  // no term
        float v[3] = {0.f, 0.f, 0.f};
        for (int k = 0; k < F.splits; ++k) {
            const float4 u = p[(size_t)k * F.n];
            const float f = xt::ex2(u.x - m);
            v[0] = fmaf(f, u.y, v[0]);
            v[1] = fmaf(f, u.z, v[1]);
            v[2] = fmaf(f, u.w, v[2]);
        }
        const float rp = F.row_pot[q][r];
        if (rp != rp) continue;  // as in grad_kernel: no exponent, no term; at +inf no shift makes the terms finite
        const float em = rp == INFINITY ? NAN : F.sign[q] * exp2f((float)((double)m + (double)F.s * (double)rp));
        for (int d = 0; d < 3; ++d) out[d] = fmaf(em, v[d], out[d]);
    }
    const size_t i = F.perm ? F.perm[r] : r;
    const float aw = F.row_w[r] * F.scale;
    for (int d = 0; d < F.D; ++d) {
        float v = aw * out[d];
        if (F.accumulate) v += F.grad[i * F.D + d];
        F.grad[i * F.D + d] = v;
    }
}

struct SoftFinish {
    const float4 *part;
    int n, splits;
    const float *row_old;
    float *row_out;
    float lam, omega;
    double eps_ln2;
    int4 *fallback;
    int *n_fallback;
};
__global__ void softmin3_finish_kernel(const __grid_constant__ SoftFinish F) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= F.n) return;
    const float4 *p = F.part + r;
    float m = kNoTerm, tot = 0.f;
    for (int k = 0; k < F.splits; ++k) m = fmaxf(m, p[(size_t)k * F.n].x);
    for (int k = 0; k < F.splits; ++k) {
        const float4 u = p[(size_t)k * F.n];
        tot += u.y * xt::ex2(u.x - m);
    }
    if (!(tot >= 0x1p-60f && tot <= 0x1p60f)) {
        F.fallback[atomicAdd(F.n_fallback, 1)] = make_int4(0, r, r / kT, 0);
        return;
    }
    const double tilde = -(double)F.lam * F.eps_ln2 * ((double)m + log2((double)tot));
    double nw = tilde;
    if (F.row_old) {
        const double old = (double)F.row_old[r];
        nw = old + (double)F.omega * (tilde - old);
    }
    F.row_out[r] = (float)nw;
}

__device__ __forceinline__ uint32_t spread3(uint32_t v) {  // bit k -> bit 3 k, 10 bits
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}
// Position on the Hilbert curve of a 2^bits grid over the points' box (J. Skilling, Programming the Hilbert curve, AIP
// Conf. Proc. 707, 2004: undo the rotations of every level from the top, then Gray-encode; the index interleaves the
// three coordinates' bits).
__global__ void hilbert_kernel(const float *x, int n, int D, const float *box, int bits, uint32_t *keys) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float ext = 0.f;
    for (int d = 0; d < D; ++d) ext = fmaxf(ext, box[64 + d] - box[d]);
    const float inv = ext > 0.f ? (float)(1 << bits) / ext : 0.f;
    uint32_t c[3] = {0u, 0u, 0u};
#pragma unroll
    for (int d = 0; d < 3; ++d)
        if (d < D) {
            const float u = (x[(size_t)i * D + d] - box[d]) * inv;
            c[d] = u > 0.f ? (uint32_t)min((int)fminf(u, 1e6f), (1 << bits) - 1) : 0u;  // also for a point that is not finite
        }
    for (uint32_t q = 1u << (bits - 1); q > 1u; q >>= 1) {
        const uint32_t low = q - 1u;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            if (c[d] & q) {
                c[0] ^= low;
            } else {
                const uint32_t u = (c[0] ^ c[d]) & low;
                c[0] ^= u;
                c[d] ^= u;
            }
        }
    }
    c[1] ^= c[0];
    c[2] ^= c[1];
    uint32_t g = 0u;
    for (uint32_t q = 1u << (bits - 1); q > 1u; q >>= 1)
        if (c[2] & q) g ^= q - 1u;
    keys[i] = (spread3(c[0] ^ g) << 2) | (spread3(c[1] ^ g) << 1) | spread3(c[2] ^ g);
}

// Order of n points along the Hilbert curve of their box (lo at d_box, hi at d_box + 64).  Five bits per axis (two sort
// passes) up to 32k points, eight (three passes) above.
int *curve_order(otgb_ctx *ctx, const std::string &tag, const float *x, int n, int D, const float *d_box) {
    cudaStream_t st = ctx_stream(ctx);
    Workspace &ws = ctx_ws(ctx);
    uint32_t *src = ws.get<uint32_t>(tag + ":k0", n), *keys = ws.get<uint32_t>(tag + ":k1", n);
    int *perm = ws.get<int>(tag + ":perm", n);
    const int bits = n <= 32768 ? 5 : 8;
    hilbert_kernel<<<(n + 255) / 256, 256, 0, st>>>(x, n, D, d_box, bits, src);
    OTGB_CHECK_LAUNCH();
    radix_sort_pairs_from(src, keys, perm, n, 3 * bits, ws.get("sort:scratch", radix_sort_scratch_bytes(n)), st);
    return perm;
}

// Fills boxes and splits, launches the sums over `parts` parts.
template <bool GRAD> void run_sums(otgb_ctx *ctx, S3Args &A, int parts, cudaStream_t st) {
    Workspace &ws = ctx_ws(ctx);
    int mx = 0;
    float4 *box[2] = {nullptr, nullptr};
    for (int q = 0; q < parts; ++q) {
        const int nt = (A.part[q].n + kT - 1) / kT;
        mx = std::max(mx, nt);
        box[q] = ws.get<float4>(q ? "s3:box1" : "s3:box0", 2 * (size_t)nt);
        A.part[q].box = box[q];
    }
    const int nblk = (A.n_rows + kT - 1) / kT;
    // about two waves of four CTAs per SM (the gradient: five); a split visits the best tile for its shift only, so at least
    // 16 tiles each (the gradient, whose tiles take longer: 4)
    const int slots = (GRAD ? 10 : 8) * ctx_sm_count(ctx), want = (slots + nblk * parts - 1) / (nblk * parts);
    A.splits = std::max(1, std::min(want, mx / (GRAD ? 4 : 16)));
    A.out = ws.get<float4>("s3:part", (size_t)parts * A.splits * A.n_rows);
    if constexpr (!GRAD) {
        A.err = ws.get<unsigned>("s3:err", 1);
        OTGB_CUDA_TRY(cudaMemsetAsync(A.err, 0, sizeof(unsigned), st));
    }
    tile_box_kernel<<<dim3((mx + 7) / 8, parts), 256, 0, st>>>(A, box[0], box[1]);
    OTGB_CHECK_LAUNCH();
    static_assert(sizeof(S3Smem) * 4 + 4096 <= 228 * 1024 && sizeof(G3Smem) * 5 + 5120 <= 228 * 1024, "CTAs per SM");
    constexpr int bytes = GRAD ? (int)sizeof(G3Smem) : (int)sizeof(S3Smem);
    const auto kernel = GRAD ? grad3_sorted_kernel : softmin3_sorted_kernel;
    static PerDevice<int> attr;
    attr.get([&] {
        OTGB_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
        return 1;
    });
    kernel<<<dim3(nblk, A.splits, parts), kT, bytes, st>>>(A);
    OTGB_CHECK_LAUNCH();
}

void check_timeout(otgb_ctx *ctx, const unsigned *err, const char *what, cudaStream_t st) {
    unsigned *h = static_cast<unsigned *>(ctx_pinned(ctx));
    OTGB_CUDA_TRY(cudaMemcpyAsync(h, err, sizeof(unsigned), cudaMemcpyDeviceToHost, st));
    OTGB_CUDA_TRY(cudaStreamSynchronize(st));
    require(*h == 0, std::string(what) + ": a bounded device wait gave up", OTGB_ETIMEOUT);
}

}  // namespace

void grad3_run(otgb_ctx *ctx, const float4 *rows, int n, int D, const Grad3Part (&part)[2], double eps, const float *row_w,
               float scale, int accumulate, const int *perm, float *grad, cudaStream_t st) {
    S3Args A;
    std::memset(&A, 0, sizeof(A));
    GradFinish F;
    std::memset(&F, 0, sizeof(F));
    A.rows = rows;
    A.n_rows = n;
    A.eps = (float)eps;
    A.s = (float)(1.4426950408889634 / eps);
    for (int q = 0; q < 2; ++q) {
        A.part[q] = S3Part{part[q].cols, part[q].pot, nullptr, part[q].n};
        F.row_pot[q] = part[q].row_pot;
        F.sign[q] = part[q].sign;
    }
    run_sums<true>(ctx, A, 2, st);
    F.part = A.out; F.n = n; F.D = D; F.splits = A.splits; F.row_w = row_w; F.perm = perm; F.s = A.s; F.scale = scale;
    F.accumulate = accumulate; F.grad = grad;
    grad3_finish_kernel<<<(n + 127) / 128, 128, 0, st>>>(F);
    OTGB_CHECK_LAUNCH();
}

void grad3_apply(otgb_ctx *ctx, const float *x, const float *alpha, int N, const float *y, const float *beta, int M, int D,
                 double eps, const float *f, const float *g, const float *a_self, float *grad) {
    cudaStream_t st = ctx_stream(ctx);
    Workspace &ws = ctx_ws(ctx);
    float *box = ws.get<float>("box", 4 * 64), *bpart = ws.get<float>("bpart", 64 * 2 * 64), *cen = ws.get<float>("cen", 64);
    bbox(x, N, D, D, box, box + 64, bpart, st);
    bbox(y, M, D, D, box + 128, box + 192, bpart, st);
    OTGB_CUDA_TRY(cudaMemsetAsync(cen, 0, 64 * sizeof(float), st));  // the coordinates as they are
    int *px = curve_order(ctx, "s3:x", x, N, D, box), *py = curve_order(ctx, "s3:y", y, M, D, box + 128);
    float4 *X = ws.get<float4>("s3:X", N), *Y = ws.get<float4>("s3:Y", M);
    float *xw = ws.get<float>("s3:xw", N), *fs = ws.get<float>("s3:f", N), *as = ws.get<float>("s3:a", N), *gs = ws.get<float>("s3:g", M);
    pack_points(x, alpha, px, N, D, cen, reinterpret_cast<float *>(X), nullptr, xw, st);
    pack_points(y, beta, py, M, D, cen, reinterpret_cast<float *>(Y), nullptr, nullptr, st);
    permute(f, px, N, fs, st);
    permute(a_self, px, N, as, st);
    permute(g, py, M, gs, st);
    const Grad3Part part[2] = {{Y, gs, M, 1.f, fs}, {X, as, N, -1.f, as}};
    grad3_run(ctx, X, N, D, part, eps, xw, 1.f, 0, px, grad, st);
    OTGB_CUDA_TRY(cudaStreamSynchronize(st));
}

void softmin3_sorted(otgb_ctx *ctx, const float *q, int n_out, const float *p, const float *w, const float *pot, int n_in,
                     int D, double eps, double lam, const float *old, double omega, float *out, const float *d_box,
                     const float *d_cen) {
    cudaStream_t st = ctx_stream(ctx);
    Workspace &ws = ctx_ws(ctx);
    float *qbox = ws.get<float>("s3:qbox", 128), *bpart = ws.get<float>("bpart", 64 * 2 * 64);
    bbox(q, n_out, D, D, qbox, qbox + 64, bpart, st);
    int *pq = curve_order(ctx, "s3:x", q, n_out, D, qbox), *pp = curve_order(ctx, "s3:y", p, n_in, D, d_box);
    float4 *R = ws.get<float4>("s3:X", n_out), *C = ws.get<float4>("s3:Y", n_in);
    float *ps = ws.get<float>("s3:g", n_in), *os = old ? ws.get<float>("s3:f", n_out) : nullptr, *res = ws.get<float>("s3:a", n_out);
    pack_points(q, nullptr, pq, n_out, D, d_cen, reinterpret_cast<float *>(R), nullptr, nullptr, st);
    pack_points(p, w, pp, n_in, D, d_cen, reinterpret_cast<float *>(C), nullptr, nullptr, st);
    permute(pot, pp, n_in, ps, st);
    if (old) permute(old, pq, n_out, os, st);
    S3Args A;
    std::memset(&A, 0, sizeof(A));
    A.rows = R;
    A.n_rows = n_out;
    A.eps = (float)eps;
    A.s = (float)(1.4426950408889634 / eps);
    A.part[0] = S3Part{C, ps, nullptr, n_in};
    run_sums<false>(ctx, A, 1, st);
    // rows whose sums are no number take the safe kernel, over all columns
    SoftminLaunch L;
    std::memset(&L, 0, sizeof(L));
    L.n_inst = 1;
    SoftminInst &I = L.inst[0];
    I.rows = reinterpret_cast<const float *>(R); I.cols = reinterpret_cast<const float *>(C);
    I.col_pot = ps; I.row_old = os; I.row_out = res;
    I.n_rows = n_out; I.n_cols = n_in; I.lam = (float)lam; I.omega = (float)omega;
    L.eps = A.eps;
    L.s = A.s;
    L.eps_ln2 = eps * 0.69314718055994530942;
    L.fallback = ws.get<int4>("sm:fb", n_out + 64);
    L.n_fallback = ws.get<int>("s3:nfb", 1);
    L.fallback_cap = n_out + 64;
    OTGB_CUDA_TRY(cudaMemsetAsync(L.n_fallback, 0, sizeof(int), st));
    const SoftFinish F{A.out, n_out, A.splits, os, res, I.lam, I.omega, L.eps_ln2, L.fallback, L.n_fallback};
    softmin3_finish_kernel<<<(n_out + 127) / 128, 128, 0, st>>>(F);
    OTGB_CHECK_LAUNCH();
    softmin_fallback_launch(L, D, st);
    unpermute(res, pq, n_out, out, st);
    check_timeout(ctx, A.err, "otgb_softmin", st);
}

}  // namespace otgb
