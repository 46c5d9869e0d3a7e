// Data-parallel primitives of the solver: reductions (bounding box, FP64
// divergence sums), exclusive scan, stable LSD radix sort, packing of the
// point clouds into the internal layout, cluster statistics.
#include <cfloat>
#include <cmath>

#include "prims.cuh"
#include "threefloat.cuh"

namespace otgb {
namespace {

constexpr int kRB = 256;  // threads per block for the reductions

// ------------------------------------------------------------------ bbox --
// V floats per load (4 when rows are whole 16-byte groups): a CTA of kBoxT threads holds kBoxT / (D / V) rows at a time, so
// consecutive threads read consecutive addresses whatever D is (one pass over the points; a pass per coordinate read
// 300k x 60 points in 329 us).  bad (optional): bit 2 when a coordinate is not finite.
constexpr int kBoxT = 1024, kBoxBlocks = 64;
template <int V>
__global__ void __launch_bounds__(kBoxT) bbox_partial_kernel(const float *x, int n, int D, int stride, float *part, int *bad) {
    // part: [gridDim.x][2*D]: lo then hi of this block
    __shared__ float red[kBoxT * V];
    const int Q = D / V, G = kBoxT / Q;  // loads per row, rows per sweep of the CTA
    const int t = threadIdx.x, g = t / Q, q = t - g * Q;
    float lo[V], hi[V];
#pragma unroll
    for (int e = 0; e < V; ++e) {
        lo[e] = FLT_MAX;
        hi[e] = -FLT_MAX;
    }
    bool fine = true;
    if (g < G) {
        const size_t step = (size_t)gridDim.x * G;
#pragma unroll 4
        for (size_t i = (size_t)blockIdx.x * G + g; i < (size_t)n; i += step) {
            float v[V];
            if constexpr (V == 4) {
                const float4 u = *reinterpret_cast<const float4 *>(x + i * stride + 4 * q);
                v[0] = u.x; v[1] = u.y; v[2] = u.z; v[3] = u.w;
            } else {
                v[0] = x[i * stride + q];
            }
#pragma unroll
            for (int e = 0; e < V; ++e) {
                lo[e] = fminf(lo[e], v[e]);
                hi[e] = fmaxf(hi[e], v[e]);
                fine = fine && isfinite(v[e]);
            }
        }
    }
    if (bad && !fine) atomicOr(bad, 2);
    for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int e = 0; e < V; ++e) red[t * V + e] = h ? hi[e] : lo[e];
        __syncthreads();
        // a warp per coordinate combines the G groups: groups lie D floats apart
        for (int d = t >> 5; d < D; d += kBoxT / 32) {
            float v = h ? -FLT_MAX : FLT_MAX;
            for (int k = t & 31; k < G; k += 32) v = h ? fmaxf(v, red[k * D + d]) : fminf(v, red[k * D + d]);
            for (int o = 16; o > 0; o >>= 1) {
                const float u = __shfl_xor_sync(0xffffffffu, v, o);
                v = h ? fmaxf(v, u) : fminf(v, u);
            }
            if ((t & 31) == 0) part[(size_t)blockIdx.x * 2 * D + h * D + d] = v;
        }
        __syncthreads();
    }
}

__global__ void bbox_final_kernel(const float *part, int nblk, int D, float *lo, float *hi) {
    const int d = threadIdx.x;
    if (d >= D) return;
    float l = FLT_MAX, h = -FLT_MAX;
#pragma unroll 16
    for (int b = 0; b < nblk; ++b) {
        l = fminf(l, part[(size_t)b * 2 * D + d]);
        h = fmaxf(h, part[(size_t)b * 2 * D + D + d]);
    }
    lo[d] = l;
    hi[d] = h;
}

__global__ void box_centre_kernel(const float *lo, const float *hi, int D, float *c) {
    const int d = threadIdx.x;
    if (d < 64) c[d] = d < D ? 0.5f * (lo[d] + hi[d]) : 0.f;
}

// Box and centre of a small input in one CTA (up to kBoxSmall values: a few microseconds, less than the launches and the
// partial results of the general form).
constexpr int kBoxSmall = 32768;
__global__ void __launch_bounds__(kBoxT) bbox_small_kernel(const float *x, int n, int D, float *c, float *box) {
    __shared__ float red[kBoxT];
    const int G = kBoxT / D, t = threadIdx.x, g = t / D, d = t - g * D;
    float lo = FLT_MAX, hi = -FLT_MAX;
    if (g < G) {
#pragma unroll 4
        for (int i = g; i < n; i += G) {
            const float v = x[(size_t)i * D + d];
            lo = fminf(lo, v);
            hi = fmaxf(hi, v);
        }
    }
    float out[2] = {0.f, 0.f};
    for (int h = 0; h < 2; ++h) {
        red[t] = h ? hi : lo;
        __syncthreads();
        for (int q = t >> 5, u = 0; q < D; q += kBoxT / 32, ++u) {
            float v = h ? -FLT_MAX : FLT_MAX;
            for (int k = t & 31; k < G; k += 32) v = h ? fmaxf(v, red[k * D + q]) : fminf(v, red[k * D + q]);
            for (int o = 16; o > 0; o >>= 1) {
                const float w = __shfl_xor_sync(0xffffffffu, v, o);
                v = h ? fmaxf(v, w) : fminf(v, w);
            }
            if ((t & 31) == 0) box[64 * h + q] = v;
            out[u] = h ? 0.5f * (out[u] + v) : v;
        }
        __syncthreads();
    }
    if ((t & 31) == 0)
        for (int q = t >> 5, u = 0; q < 64; q += kBoxT / 32, ++u) c[q] = q < D ? out[u] : 0.f;
}

// ------------------------------------------------------- FP64 sums (Eq. 6) --
// Balanced: sum_i a_i (f_i - aa_i) + sum_j b_j (g_j - bb_j).
// Unbalanced: -(rho + eps/2) [ sum_i a_i e^{-aa_i/rho} expm1(-(f_i - aa_i)/rho) + (same for b) ].
__global__ void divsum_partial_kernel(const float *wa, const float *f, const float *aa, int N, const float *wb,
                                      const float *g, const float *bb, int M, double rho, int balanced,
                                      double *part) {
    __shared__ double s[kRB];
    double acc = 0.0;
    const int total = N + M;
    for (int k = blockIdx.x * kRB + threadIdx.x; k < total; k += gridDim.x * kRB) {
        double w, p, q;
        if (k < N) { w = wa[k]; p = f[k]; q = aa[k]; }
        else { const int j = k - N; w = wb[j]; p = g[j]; q = bb[j]; }
        if (w == 0.0) continue;
        acc += balanced ? w * (p - q) : w * exp(-q / rho) * expm1(-(p - q) / rho);
    }
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int o = kRB / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = s[0];
}

__global__ void divsum_final_kernel(const double *part, int nblk, double rho, double eps, int balanced,
                                    double *out) {
    __shared__ double s[128];
    if (threadIdx.x < nblk) s[threadIdx.x] = part[threadIdx.x];
    __syncthreads();
    if (threadIdx.x != 0) return;
    double acc = 0.0;
#pragma unroll 16
    for (int b = 0; b < nblk; ++b) acc += s[b];  // fixed order: deterministic
    *out = balanced ? acc : -(rho + 0.5 * eps) * acc;
}

// ----------------------------------------------- translation of (f, g) ----
// part[b] = (sum_i a_i e^{-f_i/rho}, sum_j b_j e^{-g_j/rho}) over a grid-stride share.
__global__ void transl_partial_kernel(const float *wa, const float *f, int N, const float *wb, const float *g, int M,
                                      double rho, double2 *part) {
    __shared__ double sa[kRB], sb[kRB];
    // exp in single precision where it cannot overflow or flush (|t| < 80),
    // in double elsewhere; the sums in double
    const float inv_rho = (float)(1.0 / rho);
    auto term = [&](float w, float v) -> double {
        const float t = -v * inv_rho;
        return fabsf(t) < 80.f ? (double)(w * expf(t)) : (double)w * exp(-(double)v / rho);
    };
    double A = 0.0, B = 0.0;
    for (int i = blockIdx.x * kRB + threadIdx.x; i < N; i += gridDim.x * kRB) A += term(wa[i], f[i]);
    for (int j = blockIdx.x * kRB + threadIdx.x; j < M; j += gridDim.x * kRB) B += term(wb[j], g[j]);
    sa[threadIdx.x] = A;
    sb[threadIdx.x] = B;
    __syncthreads();
    for (int o = kRB / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) { sa[threadIdx.x] += sa[threadIdx.x + o]; sb[threadIdx.x] += sb[threadIdx.x + o]; }
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = make_double2(sa[0], sb[0]);
}

// c = (rho/2) log(A/B) from the partial sums (fixed order), then f += c, g -= c.
__global__ void transl_apply_kernel(const double2 *part, int nblk, double rho, float *f, int N, float *g, int M,
                                    double *c_out) {
    __shared__ float cs;
    if (threadIdx.x < 32) {
        double A = 0.0, B = 0.0;
        for (int b = threadIdx.x; b < nblk; b += 32) { A += part[b].x; B += part[b].y; }
        for (int o = 16; o > 0; o >>= 1) {
            A += __shfl_xor_sync(0xffffffffu, A, o);
            B += __shfl_xor_sync(0xffffffffu, B, o);
        }
        double c = (A > 0.0 && B > 0.0) ? 0.5 * rho * log(A / B) : 0.0;
        if (!isfinite(c)) c = 0.0;
        if (threadIdx.x == 0) {
            cs = (float)c;
            if (blockIdx.x == 0 && c_out) *c_out = c;
        }
    }
    __syncthreads();
    const float c = cs;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N + M; i += gridDim.x * blockDim.x) {
        if (i < N) f[i] += c;
        else g[i - N] -= c;
    }
}

// ------------------------------------------------------------------- scan --
constexpr int kScanB = 1024;

__global__ void scan_block_kernel(const int *in, int *out, int n, int *block_sums) {
    __shared__ int s[kScanB];
    const int i = blockIdx.x * kScanB + threadIdx.x;
    const int v = i < n ? in[i] : 0;
    s[threadIdx.x] = v;
    __syncthreads();
    for (int o = 1; o < kScanB; o <<= 1) {
        const int a = threadIdx.x >= o ? s[threadIdx.x - o] : 0;
        __syncthreads();
        s[threadIdx.x] += a;
        __syncthreads();
    }
    if (i < n) out[i] = s[threadIdx.x] - v;  // exclusive
    if (threadIdx.x == kScanB - 1) block_sums[blockIdx.x] = s[kScanB - 1];
}

// Up to kScanOne values in one launch, held in shared memory: every thread sums consecutive values (an odd number of them:
// no bank conflicts), one scan over the threads, reads and writes along the array.
constexpr int kScanV = 31, kScanOne = kScanB * kScanV;
__global__ void __launch_bounds__(kScanB) scan_one_kernel(const int *in, int *out, int n) {
    extern __shared__ int sv[];
    __shared__ int ws[32];
    const int per = ((n + kScanB - 1) / kScanB) | 1, i0 = min(n, (int)threadIdx.x * per), i1 = min(n, i0 + per);
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += kScanB) sv[i] = in[i];
    __syncthreads();
    int sum = 0;
    for (int i = i0; i < i1; ++i) sum += sv[i];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int x = sum;  // inclusive scan over the threads
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += u;
    }
    if (lane == 31) ws[w] = x;
    __syncthreads();
    if (w == 0) {
        int y = ws[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) y += u;
        }
        ws[lane] = y;
    }
    __syncthreads();
    int run = x - sum + (w > 0 ? ws[w - 1] : 0);
    for (int i = i0; i < i1; ++i) {
        const int v = sv[i];
        sv[i] = run;
        run += v;
    }
    __syncthreads();
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += kScanB) out[i] = sv[i];
}

__global__ void scan_add_kernel(int *out, int n, const int *block_off) {
    const int i = blockIdx.x * kScanB + threadIdx.x;
    if (i < n) out[i] += block_off[blockIdx.x];
}

// ------------------------------------------------------------- radix sort --
// Stable LSD radix sort of (key, value) pairs, 8-bit digits.  Each CTA owns a
// chunk of kChunk consecutive elements; per pass: digit histograms per chunk,
// an exclusive scan in digit-major order, then a stable scatter where each
// element's rank among equal digits of its chunk follows input order.
constexpr int kSortT = 256;
constexpr int kPerT = 4;  // 1024 keys per CTA: sorts of 16k to 131k keys then fill the GPU (8 left most of it idle)
constexpr int kChunk = kSortT * kPerT;

__global__ void radix_hist_kernel(const uint32_t *keys, int n, int shift, int *counts, int nchunks) {
    __shared__ int h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int base = blockIdx.x * kChunk;
    for (int k = 0; k < kPerT; ++k) {
        const int i = base + k * kSortT + threadIdx.x;
        if (i < n) atomicAdd(&h[(keys[i] >> shift) & 255u], 1);
    }
    __syncthreads();
    counts[(size_t)threadIdx.x * nchunks + blockIdx.x] = h[threadIdx.x];
}

__global__ void radix_scatter_kernel(const uint32_t *keys, const int *vals, int n, int shift,
                                     const int *offsets, int nchunks, uint32_t *keys_out, int *vals_out) {
    __shared__ int run[256];         // running output position per digit
    __shared__ int wc[kSortT / 32][256];  // per-warp digit counts of the current round
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    run[t] = offsets[(size_t)t * nchunks + blockIdx.x];
    const int base = blockIdx.x * kChunk;
    for (int k = 0; k < kPerT; ++k) {
        for (int q = 0; q < kSortT / 32; ++q) wc[q][t] = 0;
        __syncthreads();
        const int i = base + k * kSortT + t;
        const bool valid = i < n;
        const uint32_t key = valid ? keys[i] : 0u;
        const int dig = valid ? (int)((key >> shift) & 255u) : 256 + lane;  // unique for invalid
        const unsigned peers = __match_any_sync(0xffffffffu, dig);
        const int rank = __popc(peers & ((1u << lane) - 1u));
        if (valid && rank == 0) wc[w][dig] = __popc(peers);
        __syncthreads();
        if (valid) {
            int pos = run[dig] + rank;
            for (int q = 0; q < w; ++q) pos += wc[q][dig];
            OTGB_DCLAMP(pos, 0, n);
            keys_out[pos] = key;
            vals_out[pos] = vals ? vals[i] : i;
        }
        __syncthreads();
        int add = 0;
        for (int q = 0; q < kSortT / 32; ++q) add += wc[q][t];
        run[t] += add;
        __syncthreads();
    }
}

// ------------------------------------------------------------- packing ---
// D <= 3: out[k] = (x - c, log w) as float4 (zero-padded coordinates).
// D >  3 (pack_rows_kernel): out row k = x - c padded with zeros to D4 floats; logw[k] = log w.
__device__ __forceinline__ void pack_point(int k, const float *x, const float *w, const int *perm, int n, int D,
                                           const float *center, float *out, float *logw, float *w_sorted) {
    int i = perm ? perm[k] : k;
    OTGB_DCLAMP(i, 0, n);
    const float wi = w ? w[i] : 1.0f;
    const float lw = wi > 0.f ? logf(wi) : -INFINITY;
    float v[3] = {0.f, 0.f, 0.f};
    for (int d = 0; d < D; ++d) v[d] = x[(size_t)i * D + d] - center[d];
    reinterpret_cast<float4 *>(out)[k] = make_float4(v[0], v[1], v[2], lw);
    if (logw) logw[k] = lw;
    if (w_sorted) w_sorted[k] = wi;
}

__global__ void pack_kernel(const float *x, const float *w, const int *perm, int n, int D, const float *center,
                            float *out, float *logw, float *w_sorted) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) pack_point(k, x, w, perm, n, D, center, out, logw, w_sorted);
}

// D > 3: one thread per point and four coordinates, so that reads and writes run along the rows.
__device__ __forceinline__ void pack_quad(size_t e, const float *x, const float *w, const int *perm, int n, int D, int D4,
                                          int vec, const float *center, float *out, float *logw, float *w_sorted) {
    const int Q = D4 >> 2;
    const size_t k = e / Q;
    const int q = (int)(e - k * Q);
    if (k >= (size_t)n) return;
    int i = perm ? perm[k] : (int)k;
    OTGB_DCLAMP(i, 0, n);
    float v[4];
    if (vec) {
        const float4 u = *reinterpret_cast<const float4 *>(x + (size_t)i * D + 4 * q);
        const float4 c = *reinterpret_cast<const float4 *>(center + 4 * q);
        v[0] = u.x - c.x; v[1] = u.y - c.y; v[2] = u.z - c.z; v[3] = u.w - c.w;
    } else {
#pragma unroll
        for (int d = 0; d < 4; ++d) v[d] = 4 * q + d < D ? x[(size_t)i * D + 4 * q + d] - center[4 * q + d] : 0.f;
    }
    reinterpret_cast<float4 *>(out)[e] = make_float4(v[0], v[1], v[2], v[3]);
    if (q == 0) {
        const float wi = w ? w[i] : 1.0f;
        if (logw) logw[k] = wi > 0.f ? logf(wi) : -INFINITY;
        if (w_sorted) w_sorted[k] = wi;
    }
}

__global__ void pack_rows_kernel(const float *x, const float *w, const int *perm, int n, int D, int D4, int vec,
                                 const float *center, float *out, float *logw, float *w_sorted) {
    pack_quad((size_t)blockIdx.x * blockDim.x + threadIdx.x, x, w, perm, n, D, D4, vec, center, out, logw, w_sorted);
}

// rows and columns of one sweep: CTAs [0, split) pack the rows, the others the columns
__global__ void pack_pair_kernel(const float *q, int n_out, float *rows, const float *p, const float *w, int n_in,
                                 float *cols, float *col_logw, int D, int vec_q, int vec_p, const float *center, int split) {
    const bool r = (int)blockIdx.x < split;
    const size_t e = (size_t)(r ? blockIdx.x : blockIdx.x - split) * blockDim.x + threadIdx.x;
    if (D > 3) {
        const int D4 = (D + 3) & ~3;
        if (r) pack_quad(e, q, nullptr, nullptr, n_out, D, D4, vec_q, center, rows, nullptr, nullptr);
        else pack_quad(e, p, w, nullptr, n_in, D, D4, vec_p, center, cols, col_logw, nullptr);
    } else if (r) {
        if (e < (size_t)n_out) pack_point((int)e, q, nullptr, nullptr, n_out, D, center, rows, nullptr, nullptr);
    } else {
        if (e < (size_t)n_in) pack_point((int)e, p, w, nullptr, n_in, D, center, cols, nullptr, nullptr);
    }
}

__global__ void iota_kernel(int *v, int n) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) v[k] = k;
}

__global__ void unpermute_kernel(const float *in, const int *perm, int n, float *out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    int i = perm ? perm[k] : k;
    OTGB_DCLAMP(i, 0, n);
    out[i] = in[k];
}

__global__ void permute_kernel(const float *in, const int *perm, int n, float *out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    int i = perm ? perm[k] : k;
    OTGB_DCLAMP(i, 0, n);
    out[k] = in[i];
}

__global__ void check_weights_kernel(const float *w, int n, int *bad, double *mass_part) {
    __shared__ double s[kRB];
    double acc = 0.0;
    for (int i = blockIdx.x * kRB + threadIdx.x; i < n; i += gridDim.x * kRB) {
        const float v = w[i];
        if (!(v >= 0.f) || !(v < INFINITY)) atomicOr(bad, 1);
        else acc += v;
    }
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int o = kRB / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) mass_part[blockIdx.x] = s[0];
}

__global__ void check_points_kernel(const float *x, size_t n, int *bad) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        if (!isfinite(x[i])) atomicOr(bad, 2);
}

__global__ void absmax_kernel(const float *v, size_t n, unsigned *out) {
    float m = 0.f;
#pragma unroll 4
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) m = fmaxf(m, fabsf(v[i]));
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, __float_as_uint(m));
}

__global__ void finite_kernel(const float *v, int n, int *bad) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        if (!isfinite(v[i])) atomicOr(bad, 4);
}

// ------------------------------------------------------ cluster statistics --
// Over sorted positions [off[k], off[k+1]) of the packed points (stride floats per point): mass = sum w, centroid =
// weighted mean (plain mean when the mass is 0), radius = max distance to the centroid, ssq = sum w |x - c|^2.  Sums in at
// least FP64 accuracy, in a fixed order.
// D > 3: one CTA per cluster, thread (group g, coordinate d): a warp reads along the rows, and the points pass twice (a
// pass per coordinate with a reduction each took 380 us for 300 clusters of 1000 points; sums in FP64 290 us for 100
// clusters of 512).
constexpr int kStT = 1024, kStG = kStT / 64, kStW = kStT / 32;
__global__ void __launch_bounds__(kStT) cluster_stats_kernel(const float *pts, int stride, int D, const float *w_sorted,
                                                            const int *off, int ncl, float *cent, int cstride, float *mass,
                                                            float *radius, float *ssq) {
    __shared__ float part[3][kStG][64], mpart[3][kStG], wpart[3][kStW];
    __shared__ double vsum[64], msum;
    __shared__ float c_s[64];
    __shared__ float rmax[kStW];
    const int k = blockIdx.x;
    if (k >= ncl) return;
    const int a = off[k], b = off[k + 1];
    const int t = threadIdx.x, g = t >> 6, d = t & 63;
    // The groups' sums are combined as they are, and only 65 threads go over to FP64 (1024 of them took a third of the kernel).
    auto put = [](const ThreeFloat &f, float &hi, float &mid, float &lo) {
        hi = f.hi;
        mid = f.mid;
        lo = f.lo;
    };
    auto join = [](ThreeFloat &s, float hi, float mid, float lo) {
        s.add(hi);
        s.add_small(mid);
        s.lo += lo;
    };
    auto combine = [&] {  // vsum[d], msum from the groups' sums
        __syncthreads();
        ThreeFloat s;
        if (t < 64) {
            for (int q = 0; q < kStG; ++q) join(s, part[0][q][t], part[1][q][t], part[2][q][t]);
            vsum[t] = s.value();
        } else if (t == 64) {
            for (int q = 0; q < kStG; ++q) join(s, mpart[0][q], mpart[1][q], mpart[2][q]);
            msum = s.value();
        }
        __syncthreads();
    };
    // in double, one thread per coordinate: beyond the float range, or products that lose bits below it (rare)
    auto in_double = [&](bool weighted) {
        __syncthreads();
        double v = 0.0, m = 0.0;
        if (t < 64) {
            for (int i = a; i < b; ++i) {
                const double w = w_sorted[i];
                m += w;
                v += (weighted ? w : 1.0) * (t < D ? pts[(size_t)i * stride + t] : 0.f);
            }
            vsum[t] = v;
            if (t == 0) msum = m;
        }
        __syncthreads();
    };
    ThreeFloat acc, m;
#pragma unroll 4
    for (int i = a + g; i < b; i += kStG) {
        const float w = w_sorted[i], v = d < D ? pts[(size_t)i * stride + d] : 0.f;
        if (d == 0) m.add(w);
        acc.add_product(w, v);
    }
    put(acc, part[0][g][d], part[1][g][d], part[2][g][d]);
    if (d == 0) put(m, mpart[0][g], mpart[1][g], mpart[2][g]);
    if (__syncthreads_or(!acc.usable() || !m.usable())) in_double(true);
    else combine();
    const double mass_k = msum;
    if (!(mass_k > 0.0)) {  // uniform
        ThreeFloat plain;
        for (int i = a + g; i < b; i += kStG) plain.add(d < D ? pts[(size_t)i * stride + d] : 0.f);
        put(plain, part[0][g][d], part[1][g][d], part[2][g][d]);
        if (__syncthreads_or(!plain.usable())) in_double(false);
        else combine();
    }
    if (t < 64) c_s[t] = (float)(vsum[t] / (mass_k > 0.0 ? mass_k : (double)(b - a)));
    __syncthreads();
    // distances: a warp per point
    const int warp = t >> 5, lane = t & 31;
    const float c0 = lane < D ? c_s[lane] : 0.f, c1 = lane + 32 < D ? c_s[lane + 32] : 0.f;
    float r2 = 0.f;
    ThreeFloat wss;
    auto square = [&](int i) -> float {
        const float u = lane < D ? pts[(size_t)i * stride + lane] - c0 : 0.f;
        const float v = lane + 32 < D ? pts[(size_t)i * stride + lane + 32] - c1 : 0.f;
        float s2 = fmaf(u, u, v * v);
        for (int o = 16; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        return s2;
    };
#pragma unroll 4
    for (int i = a + warp; i < b; i += kStW) {
        const float s2 = square(i);
        r2 = fmaxf(r2, s2);
        if (ssq) wss.add_product(w_sorted[i], s2);
    }
    if (lane == 0) {
        rmax[warp] = r2;
        put(wss, wpart[0][warp], wpart[1][warp], wpart[2][warp]);
    }
    const bool bad = __syncthreads_or(!wss.usable()) != 0;
    if (bad) {  // in double
        double v = 0.0;
        for (int i = a + warp; i < b; i += kStW) v += (double)w_sorted[i] * square(i);
        if (lane == 0) vsum[warp] = v;
        __syncthreads();
    }
    if (warp == 0) {
        double ws = bad ? vsum[lane] : (double)wpart[0][lane] + ((double)wpart[1][lane] + (double)wpart[2][lane]);
        float r = rmax[lane];
        for (int o = 16; o > 0; o >>= 1) {
            ws += __shfl_xor_sync(0xffffffffu, ws, o);
            r = fmaxf(r, __shfl_xor_sync(0xffffffffu, r, o));
        }
        if (lane == 0) {
            mass[k] = (float)mass_k;
            radius[k] = sqrtf(r) * (1.0f + 1e-6f) + 1e-30f;
            if (ssq) ssq[k] = (float)ws;
        }
    }
    if (t < cstride) cent[(size_t)k * cstride + t] = t < D ? c_s[t] : 0.f;
}

// D <= 3 (float4 points): one warp per cluster.  The coarse measure is packed like the points: (centroid, log mass).
__global__ void cluster_stats3_kernel(const float4 *pts, int D, const float *w_sorted, const int *off, int ncl, float *cent,
                                      int cstride, float *mass, float *radius, float *ssq) {
    const int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (k >= ncl) return;
    const int a = off[k], b = off[k + 1];
    double v[7] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};  // mass, weighted sums, plain sums
    for (int i = a + lane; i < b; i += 32) {
        const float4 p = pts[i];
        const double w = w_sorted[i];
        v[0] += w;
        v[1] += w * p.x; v[2] += w * p.y; v[3] += w * p.z;
        v[4] += p.x; v[5] += p.y; v[6] += p.z;
    }
#pragma unroll
    for (int q = 0; q < 7; ++q)
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
    const bool pos = v[0] > 0.0;
    const double den = pos ? v[0] : (double)(b - a);
    float c[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) c[q] = q < D ? (float)((pos ? v[1 + q] : v[4 + q]) / den) : 0.f;
    float r2 = 0.f;
    double wss = 0.0;
    for (int i = a + lane; i < b; i += 32) {
        const float4 p = pts[i];
        const float u0 = p.x - c[0], u1 = p.y - c[1], u2 = p.z - c[2];
        const float s2 = fmaf(u2, u2, fmaf(u1, u1, u0 * u0));
        r2 = fmaxf(r2, s2);
        wss += (double)w_sorted[i] * s2;
    }
    for (int o = 16; o > 0; o >>= 1) {
        r2 = fmaxf(r2, __shfl_xor_sync(0xffffffffu, r2, o));
        wss += __shfl_xor_sync(0xffffffffu, wss, o);
    }
    if (lane == 0) {
        mass[k] = (float)v[0];
        radius[k] = sqrtf(r2) * (1.0f + 1e-6f) + 1e-30f;
        if (ssq) ssq[k] = (float)wss;
        for (int q = 0; q < cstride; ++q)
            cent[(size_t)k * cstride + q] = q < D ? (q == 0 ? c[0] : (q == 1 ? c[1] : c[2]))
                                                  : (q == 3 ? (pos ? (float)log(v[0]) : -INFINITY) : 0.f);
    }
}

}  // namespace

// =================================================================== host ==
void bbox(const float *x, int n, int D, int stride, float *d_lo, float *d_hi, float *d_part, cudaStream_t st, int *d_bad) {
    if (D % 4 == 0 && stride % 4 == 0 && ((uintptr_t)x & 15) == 0)
        bbox_partial_kernel<4><<<kBoxBlocks, kBoxT, 0, st>>>(x, n, D, stride, d_part, d_bad);
    else
        bbox_partial_kernel<1><<<kBoxBlocks, kBoxT, 0, st>>>(x, n, D, stride, d_part, d_bad);
    OTGB_CHECK_LAUNCH();
    bbox_final_kernel<<<1, 64, 0, st>>>(d_part, kBoxBlocks, D, d_lo, d_hi);
    OTGB_CHECK_LAUNCH();
}

void box_centre(const float *lo, const float *hi, int D, float *c, cudaStream_t st) {
    box_centre_kernel<<<1, 64, 0, st>>>(lo, hi, D, c);
    OTGB_CHECK_LAUNCH();
}

void bbox_centre(const float *x, int n, int D, float *d_centre, float *d_box, float *d_part, cudaStream_t st) {
    if ((size_t)n * D <= kBoxSmall) {
        bbox_small_kernel<<<1, kBoxT, 0, st>>>(x, n, D, d_centre, d_box);
        OTGB_CHECK_LAUNCH();
        return;
    }
    bbox(x, n, D, D, d_box, d_box + 64, d_part, st);
    box_centre(d_box, d_box + 64, D, d_centre, st);
}

void divergence_sum(const float *wa, const float *f, const float *aa, int N, const float *wb, const float *g,
                    const float *bb, int M, double eps, double rho, double *d_out, double *d_part,
                    cudaStream_t st) {
    const int nblk = 128;
    const int balanced = std::isinf(rho) ? 1 : 0;
    divsum_partial_kernel<<<nblk, kRB, 0, st>>>(wa, f, aa, N, wb, g, bb, M, rho, balanced, d_part);
    OTGB_CHECK_LAUNCH();
    divsum_final_kernel<<<1, 128, 0, st>>>(d_part, nblk, rho, eps, balanced, d_out);
    OTGB_CHECK_LAUNCH();
}

void translate_duals(const float *wa, float *f, int N, const float *wb, float *g, int M, double rho, double2 *d_part,
                     double *d_c, cudaStream_t st) {
    const int nblk = 64;  // d_part holds 64 partials
    transl_partial_kernel<<<nblk, kRB, 0, st>>>(wa, f, N, wb, g, M, rho, d_part);
    OTGB_CHECK_LAUNCH();
    transl_apply_kernel<<<128, 256, 0, st>>>(d_part, nblk, rho, f, N, g, M, d_c);
    OTGB_CHECK_LAUNCH();
}

size_t scan_scratch_ints(int n) {
    const int nb = (n + kScanB - 1) / kScanB;
    return (size_t)nb + scan_scratch_ints_level(nb);
}
size_t scan_scratch_ints_level(int nb) {
    if (nb <= 1) return 2;
    return scan_scratch_ints(nb) + (size_t)nb;
}

void exclusive_scan(const int *in, int *out, int n, int *scratch, cudaStream_t st) {
    if (n <= 0) return;
    if (n <= kScanOne) {
        static PerDevice<int> attr;
        attr.get([] {
            OTGB_CUDA_TRY(cudaFuncSetAttribute(scan_one_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               kScanOne * (int)sizeof(int)));
            return 1;
        });
        scan_one_kernel<<<1, kScanB, n * sizeof(int), st>>>(in, out, n);
        OTGB_CHECK_LAUNCH();
        return;
    }
    const int nb = (n + kScanB - 1) / kScanB;
    int *bsum = scratch;
    scan_block_kernel<<<nb, kScanB, 0, st>>>(in, out, n, bsum);
    OTGB_CHECK_LAUNCH();
    if (nb > 1) {
        int *boff = scratch + nb;
        exclusive_scan(bsum, boff, nb, boff + nb, st);
        scan_add_kernel<<<nb, kScanB, 0, st>>>(out, n, boff);
        OTGB_CHECK_LAUNCH();
    }
}

size_t radix_sort_scratch_bytes(int n) {
    const int nchunks = (n + kChunk - 1) / kChunk;
    const size_t cnt = (size_t)256 * nchunks;
    return sizeof(int) * (2 * cnt + scan_scratch_ints((int)cnt) + 64) + (sizeof(uint32_t) + sizeof(int)) * (size_t)n +
           256;
}

void radix_sort_pairs_from(const uint32_t *src, uint32_t *keys, int *vals, int n, int nbits, void *scratch, cudaStream_t st) {
    if (n <= 1 || nbits <= 0) {  // one key, or keys all equal: identity permutation
        if (n >= 1 && src != keys) OTGB_CUDA_TRY(cudaMemcpyAsync(keys, src, sizeof(uint32_t) * n, cudaMemcpyDeviceToDevice, st));
        if (n >= 1) iota(vals, n, st);
        return;
    }
    const int nchunks = (n + kChunk - 1) / kChunk;
    const size_t cnt = (size_t)256 * nchunks;
    int *counts = static_cast<int *>(scratch);
    int *offs = counts + cnt;
    int *scan_scr = offs + cnt;
    uint8_t *p = reinterpret_cast<uint8_t *>(scan_scr + scan_scratch_ints((int)cnt) + 64);
    uint32_t *k2 = reinterpret_cast<uint32_t *>(p);
    int *v2 = reinterpret_cast<int *>(k2 + n);
    const int passes = (nbits + 7) / 8;
    // the passes alternate between (keys, vals) and the scratch pair so that the last one writes (keys, vals); the first
    // reads src, which must not be what it writes
    const uint32_t *kin = src;
    const int *vin = nullptr;  // first pass: values are the input positions
    bool to_keys = passes % 2 == 1;
    if (to_keys && src == keys) {
        OTGB_CUDA_TRY(cudaMemcpyAsync(k2, src, sizeof(uint32_t) * n, cudaMemcpyDeviceToDevice, st));
        kin = k2;
    }
    for (int ps = 0; ps < passes; ++ps) {
        uint32_t *kout = to_keys ? keys : k2;
        int *vout = to_keys ? vals : v2;
        radix_hist_kernel<<<nchunks, kSortT, 0, st>>>(kin, n, 8 * ps, counts, nchunks);
        OTGB_CHECK_LAUNCH();
        exclusive_scan(counts, offs, (int)cnt, scan_scr, st);
        radix_scatter_kernel<<<nchunks, kSortT, 0, st>>>(kin, vin, n, 8 * ps, offs, nchunks, kout, vout);
        OTGB_CHECK_LAUNCH();
        kin = kout;
        vin = vout;
        to_keys = !to_keys;
    }
}

void radix_sort_pairs(uint32_t *keys, int *vals, int n, int nbits, void *scratch, cudaStream_t st) {
    radix_sort_pairs_from(keys, keys, vals, n, nbits, scratch, st);
}

void iota(int *v, int n, cudaStream_t st) {
    iota_kernel<<<(n + 255) / 256, 256, 0, st>>>(v, n);
    OTGB_CHECK_LAUNCH();
}

void pack_points(const float *x, const float *w, const int *perm, int n, int D, const float *d_center, float *out,
                 float *logw, float *w_sorted, cudaStream_t st) {
    if (D > 3) {
        const int D4 = (D + 3) & ~3;
        const int vec = D % 4 == 0 && ((uintptr_t)x & 15) == 0 && ((uintptr_t)d_center & 15) == 0;
        const size_t tot = (size_t)n * (D4 >> 2);
        pack_rows_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(x, w, perm, n, D, D4, vec, d_center, out, logw, w_sorted);
    } else {
        pack_kernel<<<(n + 255) / 256, 256, 0, st>>>(x, w, perm, n, D, d_center, out, logw, w_sorted);
    }
    OTGB_CHECK_LAUNCH();
}

void pack_pair(const float *q, int n_out, float *rows, const float *p, const float *w, int n_in, float *cols, float *col_logw,
               int D, const float *d_center, cudaStream_t st) {
    const size_t per = D > 3 ? (size_t)(((D + 3) & ~3) >> 2) : 1;
    const unsigned gr = (unsigned)((n_out * per + 255) / 256), gc = (unsigned)((n_in * per + 255) / 256);
    const bool v4 = D % 4 == 0 && ((uintptr_t)d_center & 15) == 0;
    pack_pair_kernel<<<gr + gc, 256, 0, st>>>(q, n_out, rows, p, w, n_in, cols, col_logw, D, v4 && ((uintptr_t)q & 15) == 0,
                                              v4 && ((uintptr_t)p & 15) == 0, d_center, (int)gr);
    OTGB_CHECK_LAUNCH();
}

void unpermute(const float *in, const int *perm, int n, float *out, cudaStream_t st) {
    unpermute_kernel<<<(n + 255) / 256, 256, 0, st>>>(in, perm, n, out);
    OTGB_CHECK_LAUNCH();
}

void permute(const float *in, const int *perm, int n, float *out, cudaStream_t st) {
    permute_kernel<<<(n + 255) / 256, 256, 0, st>>>(in, perm, n, out);
    OTGB_CHECK_LAUNCH();
}

void check_weights(const float *w, int n, int *d_bad, double *d_mass_part, cudaStream_t st) {
    check_weights_kernel<<<64, kRB, 0, st>>>(w, n, d_bad, d_mass_part);
    OTGB_CHECK_LAUNCH();
}

void check_points(const float *x, size_t n, int *d_bad, cudaStream_t st) {
    check_points_kernel<<<256, 256, 0, st>>>(x, n, d_bad);
    OTGB_CHECK_LAUNCH();
}

void absmax(const float *v, size_t n, unsigned *d_out, cudaStream_t st) {
    absmax_kernel<<<152, 256, 0, st>>>(v, n, d_out);
    OTGB_CHECK_LAUNCH();
}

void check_finite(const float *v, int n, int *d_bad, cudaStream_t st) {
    finite_kernel<<<128, 256, 0, st>>>(v, n, d_bad);
    OTGB_CHECK_LAUNCH();
}

void cluster_stats(const float *pts, int stride, int D, const float *w_sorted, const int *off, int ncl, float *cent,
                   int cstride, float *mass, float *radius, float *ssq, cudaStream_t st) {
    if (ncl <= 0) return;
    if (D <= 3) {
        require(stride == 4, "cluster_stats: D <= 3 points are float4", OTGB_EINTERNAL);
        cluster_stats3_kernel<<<(ncl + 7) / 8, 256, 0, st>>>(reinterpret_cast<const float4 *>(pts), D, w_sorted, off, ncl,
                                                             cent, cstride, mass, radius, ssq);
    } else {
        cluster_stats_kernel<<<ncl, kStT, 0, st>>>(pts, stride, D, w_sorted, off, ncl, cent, cstride, mass, radius, ssq);
    }
    OTGB_CHECK_LAUNCH();
}

}  // namespace otgb
