// Weighted Lloyd K-means, the "simple K-means" coarse subsampling of
// Section 2: seeded sample of K distinct points as initial centroids, then
// rounds of nearest-centroid assignment (lowest index on ties) and
// weighted-mean update (an empty cluster keeps its centroid), a final
// assignment, and a stable sort of the points by cluster.
#include <cfloat>
#include <cmath>
#include <unordered_set>
#include <vector>

#include "kmeans.cuh"
#include "prims.cuh"
#include "solver.cuh"

namespace otgb {
namespace {

constexpr int kAT = 256;   // threads
constexpr int kAR = 128;   // points per CTA
constexpr int kAC = 64;    // centroids per tile

// Nearest centroid by argmin_k (|c_k|^2 - 2 x.c_k): each thread keeps 8 points x 4 centroids of dot products,
// register-tiled like a GEMM.  The four centroids go in pairs through packed f32x2 FMAs (each half is the scalar chain
// over the coordinates, so the result does not change), the point operand is stored twice per value so that one
// 16-byte load feeds two packed operands; the next centroid tile is fetched into registers while this one is
// multiplied, and |c_k|^2 comes from a launch of its own (64 threads computing it per tile left the others waiting).
// Bound: FP32 FMA, n K D lane operations.
struct AssignSmem {
    float2 xs[64][kAR];         // (v, v)
    float cs[2][64][kAC];
    float cn[2][kAC];
    float bd[16][kAR];
    int bk[16][kAR];
};

__device__ __forceinline__ unsigned long long fma2k(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__global__ void centroid_norm_kernel(const float *cent, int K, int D4, float *cn) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= K) return;
    const float4 *c4 = reinterpret_cast<const float4 *>(cent + (size_t)k * D4);
    float acc = 0.f;
#pragma unroll 8
    for (int q = 0; q < D4 / 4; ++q) {
        const float4 v = c4[q];
        acc = fmaf(v.w, v.w, fmaf(v.z, v.z, fmaf(v.y, v.y, fmaf(v.x, v.x, acc))));
    }
    cn[k] = acc;
}

__global__ void __launch_bounds__(kAT, 2) kmeans_assign_kernel(const float *x, int n, int D, int D4, const float *cent,
                                                               const float *cnorm, int K, int *labels) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    AssignSmem &S = *reinterpret_cast<AssignSmem *>(smem_raw);
    const int t = threadIdx.x, r0 = blockIdx.x * kAR;
    for (int e = t; e < kAR * D4; e += kAT) {
        const int r = e / D4, k = e - r * D4;
        const float v = (r0 + r < n && k < D) ? x[(size_t)(r0 + r) * D + k] : 0.f;
        S.xs[k][r] = make_float2(v, v);
    }
    // centroid tile: thread (centroid t % 64, quads t / 64, + 4, ..) moves up to four 16-byte pieces
    const int cc = t & 63, q0 = t >> 6, Q = D4 >> 2;
    float4 pre[4];
    float pn = INFINITY;
    auto fetch = [&](int c0) {
        const bool in = c0 + cc < K;
        const float4 *src = reinterpret_cast<const float4 *>(cent + (size_t)(in ? c0 + cc : 0) * D4);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int q = q0 + 4 * u;
            pre[u] = in && q < Q ? src[q] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if (q0 == 0) pn = in ? cnorm[c0 + cc] : INFINITY;
    };
    auto store = [&](int buf) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int q = q0 + 4 * u;
            if (q < Q) {
                S.cs[buf][4 * q][cc] = pre[u].x;
                S.cs[buf][4 * q + 1][cc] = pre[u].y;
                S.cs[buf][4 * q + 2][cc] = pre[u].z;
                S.cs[buf][4 * q + 3][cc] = pre[u].w;
            }
        }
        if (q0 == 0) S.cn[buf][cc] = pn;
    };
    const int tr = t >> 4, tc = t & 15;
    float best[8];
    int bidx[8];
#pragma unroll
    // cluster 0 until a distance is finite: a point that is not finite, or whose squares overflow, keeps it, so that every
    // label indexes a cluster
    for (int i = 0; i < 8; ++i) { best[i] = INFINITY; bidx[i] = 0; }
    fetch(0);
    store(0);
    __syncthreads();
    int buf = 0;
    for (int c0 = 0; c0 < K; c0 += kAC, buf ^= 1) {
        if (c0 + kAC < K) fetch(c0 + kAC);
        unsigned long long acc[8][2];
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i][0] = acc[i][1] = 0ull;
#pragma unroll 4
        for (int k = 0; k < D4; ++k) {
            const ulonglong2 cv = *reinterpret_cast<const ulonglong2 *>(&S.cs[buf][k][tc * 4]);
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const ulonglong2 xv = *reinterpret_cast<const ulonglong2 *>(&S.xs[k][tr * 8 + 2 * h]);
                acc[2 * h][0] = fma2k(xv.x, cv.x, acc[2 * h][0]);
                acc[2 * h][1] = fma2k(xv.x, cv.y, acc[2 * h][1]);
                acc[2 * h + 1][0] = fma2k(xv.y, cv.x, acc[2 * h + 1][0]);
                acc[2 * h + 1][1] = fma2k(xv.y, cv.y, acc[2 * h + 1][1]);
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = c0 + tc * 4 + j;
            const float cn = S.cn[buf][tc * 4 + j];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const unsigned long long w = acc[i][j >> 1];
                const float dot = __uint_as_float((j & 1) ? (unsigned)(w >> 32) : (unsigned)w);
                const float d = fmaf(-2.f, dot, cn);
                if (d < best[i] || (d == best[i] && c < bidx[i])) { best[i] = d; bidx[i] = c; }
            }
        }
        // the other buffer was read before the last barrier
        if (c0 + kAC < K) store(buf ^ 1);
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) { S.bd[tc][tr * 8 + i] = best[i]; S.bk[tc][tr * 8 + i] = bidx[i]; }
    __syncthreads();
    if (t < kAR && r0 + t < n) {
        float b = S.bd[0][t];
        int k = S.bk[0][t];
        for (int q = 1; q < 16; ++q) {
            const float d = S.bd[q][t];
            const int kk = S.bk[q][t];
            if (d < b || (d == b && kk < k)) { b = d; k = kk; }
        }
        labels[r0 + t] = k;
    }
}

// every s-th row (and weight) of x: out row i = x row i s
__global__ void strided_rows_kernel(const float *x, const float *w, int D, int s, int ni, float *out, float *wout) {
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (size_t)ni * D) return;
    const size_t i = e / D, d = e - i * D;
    out[e] = x[i * (size_t)s * D + d];
    if (w && d == 0) wout[i] = w[i * (size_t)s];
}

// Weighted mean of each cluster from the points sorted by cluster: CTA k sums
// its cluster's rows in a fixed order (4 interleaved row groups, combined in a
// fixed tree), so the centroids do not depend on scheduling.  An empty cluster
// keeps its centroid.
__global__ void kmeans_segment_mean_kernel(const float *x, const float *w, int D, int D4, const int *perm,
                                           const int *off, float *cent) {
    __shared__ float ps[4][64];
    __shared__ float pm[4];
    const int k = blockIdx.x, t = threadIdx.x, d = t & 63, g = t >> 6;
    const int a = off[k], b = off[k + 1];
    float s = 0.f, m = 0.f;
    // eight rows' indices, then their values, in flight at once; summed in order
    for (int i = a + g; i < b; i += 32) {
        int src[8];
        float wi[8], v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) src[u] = i + 4 * u < b ? perm[i + 4 * u] : -1;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            wi[u] = src[u] >= 0 ? (w ? w[src[u]] : 1.f) : 0.f;
            v[u] = src[u] >= 0 && d < D ? x[(size_t)src[u] * D + d] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (src[u] >= 0) {
                s = fmaf(wi[u], v[u], s);
                m += wi[u];
            }
    }
    ps[g][d] = s;
    if (d == 0) pm[g] = m;
    __syncthreads();
    if (g == 0 && d < D) {
        const float S = (ps[0][d] + ps[1][d]) + (ps[2][d] + ps[3][d]);
        const float M = (pm[0] + pm[1]) + (pm[2] + pm[3]);
        if (M > 0.f) cent[(size_t)k * D4 + d] = S / M;
    }
}

__global__ void gather_rows_kernel(const float *x, int D, const int *idx, int K, float *out, int D4) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= K * D4) return;
    const int k = e / D4, d = e - k * D4;
    out[e] = d < D ? x[(size_t)idx[k] * D + d] : 0.f;
}

__global__ void copy_rows_kernel(const float *src, int D, int K, float *out, int D4) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= K * D4) return;
    const int k = e / D4, d = e - k * D4;
    out[e] = d < D ? src[(size_t)k * D + d] : 0.f;
}

// offsets[k] = first sorted position with cluster >= k, k <= K
__global__ void offsets_kernel(const uint32_t *keys, int m, int K, int *offsets) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= m) return;
    const int cur = (int)keys[j], prev = j > 0 ? (int)keys[j - 1] : -1;
    for (int k = prev + 1; k <= cur; ++k) offsets[k] = j;
    if (j == m - 1)
        for (int k = cur + 1; k <= K; ++k) offsets[k] = m;
}

// Stable sort by cluster and offsets of all K clusters (empty ones included) of the first m points of the buffers.
struct LabelSort {
    uint32_t *keys;
    void *scr;
    int K, bits = 0;
    LabelSort(otgb_ctx *ctx, const std::string &tag, int n, int K_) : K(K_) {
        Workspace &ws = ctx_ws(ctx);
        keys = ws.get<uint32_t>(tag + ":keys", n);
        while ((1 << bits) < K) ++bits;
        scr = ws.get("sort:scratch", radix_sort_scratch_bytes(n));
    }
    void run(const int *labels, int m, int *perm, int *offsets, cudaStream_t st) {
        radix_sort_pairs_from(reinterpret_cast<const uint32_t *>(labels), keys, perm, m, bits, scr, st);
        offsets_kernel<<<(m + 255) / 256, 256, 0, st>>>(keys, m, K, offsets);
        OTGB_CHECK_LAUNCH();
    }
};

uint64_t splitmix64(uint64_t &s) {
    uint64_t z = (s += 0x9e3779b97f4a7c15ull);
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

}  // namespace

// K distinct indices in [0, n) by Floyd's sampling with a splitmix64 stream.
std::vector<int> sample_distinct(int n, int K, unsigned long long seed) {
    std::vector<int> out;
    std::unordered_set<int> used;
    uint64_t s = seed;
    for (int j = n - K; j < n; ++j) {
        const int t = (int)(splitmix64(s) % (uint64_t)(j + 1));
        if (used.count(t)) { used.insert(j); out.push_back(j); }
        else { used.insert(t); out.push_back(t); }
    }
    return out;
}

void kmeans_assign(const float *x, int n, int D, const float *cent, float *cnorm, int K, int *labels, cudaStream_t st) {
    const int D4 = (D + 3) & ~3;
    centroid_norm_kernel<<<(K + 127) / 128, 128, 0, st>>>(cent, K, D4, cnorm);
    OTGB_CHECK_LAUNCH();
    static PerDevice<int> attr;
    attr.get([] {
        OTGB_CUDA_TRY(cudaFuncSetAttribute(kmeans_assign_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)sizeof(AssignSmem)));
        return 1;
    });
    kmeans_assign_kernel<<<(n + kAR - 1) / kAR, kAT, sizeof(AssignSmem), st>>>(x, n, D, D4, cent, cnorm, K, labels);
    OTGB_CHECK_LAUNCH();
}

KmeansResult kmeans(otgb_ctx *ctx, const std::string &tag, const float *x, const float *w, int n, int D, int K,
                    int iters, unsigned long long seed, const float *init, int sample_max) {
    cudaStream_t st = ctx_stream(ctx);
    Workspace &ws = ctx_ws(ctx);
    const int D4 = (D + 3) & ~3;
    KmeansResult r;
    r.cstride = D4;
    r.K = K;
    r.centroids = ws.get<float>(tag + ":cent", (size_t)K * D4);
    r.labels = ws.get<int>(tag + ":lab", n);
    r.perm = ws.get<int>(tag + ":perm", n);
    r.offsets = ws.get<int>(tag + ":off", K + 1);
    float *cnorm = ws.get<float>(tag + ":cn", K);
    // the points the Lloyd iterations run on: all of them, or every s-th
    const float *xi = x, *wi = w;
    int ni = n;
    if (sample_max > 0 && n > sample_max) {
        const int sstep = (n + sample_max - 1) / sample_max;
        ni = (n + sstep - 1) / sstep;
        float *xs = ws.get<float>(tag + ":xs", (size_t)ni * D);
        float *wsub = w ? ws.get<float>(tag + ":ws", ni) : nullptr;
        strided_rows_kernel<<<(unsigned)(((size_t)ni * D + 255) / 256), 256, 0, st>>>(x, w, D, sstep, ni, xs, wsub);
        OTGB_CHECK_LAUNCH();
        xi = xs;
        wi = wsub;
    }
    if (init) {
        copy_rows_kernel<<<(K * D4 + 255) / 256, 256, 0, st>>>(init, D, K, r.centroids, D4);
        OTGB_CHECK_LAUNCH();
    } else {
        std::vector<int> idx = sample_distinct(ni, K, seed);
        int *d_idx = ws.get<int>(tag + ":idx", K);
        OTGB_CUDA_TRY(cudaMemcpyAsync(d_idx, idx.data(), sizeof(int) * K, cudaMemcpyHostToDevice, st));
        gather_rows_kernel<<<(K * D4 + 255) / 256, 256, 0, st>>>(xi, D, d_idx, K, r.centroids, D4);
        OTGB_CHECK_LAUNCH();
        OTGB_CUDA_TRY(cudaStreamSynchronize(st));  // idx is host memory about to go out of scope
    }
    LabelSort sorter(ctx, tag, n, K);
    auto sort_by_label = [&](int m) { sorter.run(r.labels, m, r.perm, r.offsets, st); };
    for (int it = 0; it < iters; ++it) {
        kmeans_assign(xi, ni, D, r.centroids, cnorm, K, r.labels, st);
        sort_by_label(ni);
        kmeans_segment_mean_kernel<<<K, 256, 0, st>>>(xi, wi, D, D4, r.perm, r.offsets, r.centroids);
        OTGB_CHECK_LAUNCH();
    }
    kmeans_assign(x, n, D, r.centroids, cnorm, K, r.labels, st);
    sort_by_label(n);
    r.sorted_keys = sorter.keys;
    return r;
}

}  // namespace otgb
