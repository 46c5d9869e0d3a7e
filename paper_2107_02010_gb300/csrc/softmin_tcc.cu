// Cluster-tiled tensor-core form of the softmin sweep (D4 <= 60, coarse-to-fine solves): the column operand is
// prepared once per solve and the CUDA cores evaluate only ex2 and the sum.
//
// In the kernel truncation of Section 2 every row block walks the columns of its kept column clusters J.
// Centring the pair at the column cluster's centre c_J instead of at the row block's centre,
//   -|x_i - y_j|^2 / 2 = (x_i - c_J) . yh_j - |x_i - c_J|^2 / 2 - |yh_j|^2 / 2,   yh_j = y_j - c_J,
// makes the column operand yh_j independent of the row block: it is split into BF16 pieces once per solve and
// stored in global memory as ready tiles of 128 columns (tcc_build), so the kernel brings each tile with one bulk
// TMA copy.  The rest of the exponent rides in the last K slots (xtile.cuh):
//   H_j  = s (eps log w_j + pot_j - |yh_j|^2 / 2) on the column side (rewritten every step by tcc_update),
//   R_iJ = -s |x_i - c_J|^2 / 2 - M_i on the row side, M_i = -s old_i / lam,
// so that the accumulator holds e_ij = (exponent of the pair in base 2) - M_i, and the finish takes
// M_i + log2 sum_j 2^e_ij in double.  The row operand is restaged once per kept cluster of the block.
//
// Two pieces per operand (NP = 2) are the reduced-precision form (OTGB_TC_BF16X3); three (NP = 3) hold 24 bits and
// are the float32 form of coarse-to-fine solves with k-means clusters: 6 x 2 K tensor flops per pair, where the
// CUDA-core form (softmin_gen_kernel) needs D + 2 FP32 operations at a fiftieth of the rate.
// Bound: the tensor pipe, 1910.7 TFLOP/s (measured) / (2 K x products) = 2.49e12 (NP = 3) and 4.98e12 (NP = 2)
// pairs/s at K = 64.  Measured on the 60-D fiber bundles (300k and 1M per side): NP = 3 2.30e12 pairs/s = 92 %, where
// softmin_gen_kernel has 3.9e11 (a solve of 300k per side 379 -> 71 ms); NP = 2 3.76e12 = 75 %, where the form with
// the row operand in shared memory, one warp group for everything and two accumulators had 2.9e12.  Error of one
// step of NP = 3 against FP64, geometric mean over D = 5 .. 60: 1.07e-7 of the duals, softmin_gen_kernel 1.28e-7.
//
// One CTA owns a block of at most 128 rows; two CTAs share an SM (256 tensor-memory columns and about 97 KB of
// shared memory each), so that the MMAs of one run while the other sums.  Warps 0-3: one row per thread -- the row
// operand into tensor memory, the sums; warp 4: one lane issues the bulk copies; warp 5: one lane issues the MMAs.
// No CTA barrier after the setup: the roles hand tiles over through mbarriers.  Every wait is bounded; a timeout
// sets an error word and the kernel still releases its tensor memory.
#include <cfloat>
#include <cmath>

#include "otgb_internal.cuh"
#include "xtile.cuh"

namespace otgb {
namespace {

constexpr int kN = xt::kCols;
constexpr int kMaxWords = kTccMaxWords;
constexpr int kThreads = 192;
struct TccCtl {
    unsigned words[kMaxWords];  // kept column clusters of this block
    unsigned long long full[xt::kMaxStages], empty[xt::kMaxStages], acc_full, acc_free, a_ready[2], drain;
    uint32_t tslot;
    int ncols;
    int abort;
};

template <int NP, int K>
__global__ void __launch_bounds__(kThreads, 2) softmin_tcc_kernel(const __grid_constant__ SoftminLaunch L, int D4) {
    using G = xt::Geom<NP, K>;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *tiles_s = smem_raw;  // stages
    TccCtl &S = *reinterpret_cast<TccCtl *>(smem_raw + G::stages * G::tile);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    int4 item = L.items[blockIdx.x];
    OTGB_DCLAMP(item.x, 0, L.n_inst);
    const SoftminInst &I = L.inst[item.x];
    const int blk = item.y;
    int r0 = I.blk_row0[blk], r1 = I.blk_row0[blk + 1];
    OTGB_DCLAMP(r0, 0, I.n_rows + 1);
    OTGB_DCLAMP(r1, r0, min(I.n_rows, r0 + xt::kRows) + 1);
    const int nr = r1 - r0;
    const float s = L.s;
    const int nwords = L.tcc_nwords;
    volatile int *abort = &S.abort;

    // ---- kept column clusters of this block: union of its row clusters' keep bits
    const int cl0 = I.tcc_blk_cl[2 * blk], cl1 = I.tcc_blk_cl[2 * blk + 1];
    if (t == 0) {
        S.ncols = 0;
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
    __syncthreads();
    int ncols = 0;
    for (int w = t; w < nwords; w += kThreads) {
        unsigned u = 0u;
        for (int c = cl0; c < cl1; ++c) u |= I.tcc_bits[(size_t)c * nwords + w];
        S.words[w] = u;
        while (u) {
            const int J = w * 32 + __ffs(u) - 1;
            u &= u - 1u;
            ncols += I.tcc_coff[J + 1] - I.tcc_coff[J];
        }
    }
    if (ncols) atomicAdd(&S.ncols, ncols);

    // ---- this thread's row (its coordinates stay in registers): M_i = -s old_i / lam
    const bool valid = t < nr;
    float Mi = 0.f;
    float x[K - 4];
    if (warp < 4) {
        const float4 *xr4 = reinterpret_cast<const float4 *>(I.rows + (size_t)(r0 + (valid ? t : 0)) * D4);
#pragma unroll
        for (int q = 0; q < K / 4 - 1; ++q) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (valid && 4 * q < D4) v = xr4[q];
            x[4 * q] = v.x;
            x[4 * q + 1] = v.y;
            x[4 * q + 2] = v.z;
            x[4 * q + 3] = v.w;
        }
        if (valid) Mi = (float)(-(double)s * (double)I.row_old[r0 + t] / (double)I.lam);
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = S.tslot;
    const int *tile0 = I.tcc_tile0;
    float tot = 0.f;
    bool ok = true;

    if (warp == 4) {
        // ---------------------------------------------------------- column tiles
        if (lane == 0) {
            xt::TileIt it;
            int k = 0;
            while (xt::tile_next(it, S.words, nwords, tile0)) {
                const int st = k % G::stages;
                if (k >= G::stages && !xt::wait(&S.empty[st], (uint32_t)((k / G::stages - 1) & 1), abort)) {
                    *abort = 1;
                    break;
                }
                xt::tma_load(tiles_s + st * G::tile, I.tcc_tiles + (size_t)it.g * G::tile, (uint32_t)G::tile, &S.full[st]);
                ++k;
            }
            // nothing in flight at exit: the last copy into each stage has landed
            for (int q = max(0, k - G::stages); q < k; ++q)
                if (!tc::mbar_wait(&S.full[q % G::stages], (uint32_t)((q / G::stages) & 1))) *abort = 1;
        }
        __syncwarp();
    } else if (warp == 5) {
        // ------------------------------------------------------------------ MMAs
        if (lane == 0) {
            xt::TileIt it;
            int k = 0, aJ = -1, na = 0;  // na: row operands taken so far
            while (xt::tile_next(it, S.words, nwords, tile0)) {
                const int st = k % G::stages;
                if (it.J != aJ) {
                    const int ab = na % G::abuf;
                    if (!xt::wait(&S.a_ready[ab], (uint32_t)((na / G::abuf) & 1), abort)) {
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
                const uint32_t a = tmem + kN + (uint32_t)(((na - 1) % G::abuf) * NP * (K / 2));
                xt::issue<NP, K>(tmem, a, tc::smem_u32(tiles_s + st * G::tile), k & 1);
                tc::commit(&S.empty[st]);
                tc::commit(&S.acc_full);
                ++k;
            }
            // nothing in flight at exit: every MMA issued completed
            tc::commit(&S.drain);
            if (!tc::mbar_wait(&S.drain, 0)) ok = false;
            if (!ok) *abort = 1;
        }
        __syncwarp();
    } else {
        // --------------------------------------------------- row operands and sums
        const uint32_t lanes = tmem + ((uint32_t)(warp * 32) << 16);
        int na = 0;  // row operands staged so far
        auto stage = [&](int J) {
            const uint32_t a = lanes + kN + (uint32_t)((na % G::abuf) * NP * (K / 2));
            xt::stage_row<NP, K>(x, D4, I.tcc_ccen + (size_t)J * D4, s, Mi, valid, a);
            xt::st_wait();
            tc::fence_before();
            xt::arrive(&S.a_ready[na % G::abuf]);
            ++na;
        };
        xt::TileIt it;
        bool have = xt::tile_next(it, S.words, nwords, tile0);
        if (have) stage(it.J);
        for (int k = 0; have; ++k) {
            xt::TileIt nx = it;
            const bool more = xt::tile_next(nx, S.words, nwords, tile0);
            const bool fresh = more && nx.J != it.J;
            // the other row operand belongs to an earlier cluster, whose MMAs are complete: tile k - 1's are
            if (G::abuf == 2 && fresh) stage(nx.J);
            ok = __all_sync(0xffffffffu, xt::wait(&S.acc_full, (uint32_t)(k & 1), abort));
            if (!ok) {  // tensor-memory loads are warp-collective
                *abort = 1;
                break;
            }
            tc::fence_after();
            tot = xt::sum_row(lanes, tot, [&] {
                tc::fence_before();
                xt::arrive(&S.acc_free);
            });
            if (G::abuf == 1 && fresh) stage(nx.J);  // tile k was the cluster's last: its MMAs are complete
            it = nx;
            have = more;
        }
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    ok = S.abort == 0;
    if (!ok && t == 0 && L.tc_err) atomicOr(L.tc_err, 1u);
    if (warp == 5) tc::tmem_dealloc(tmem, xt::kTmemCols);

    if (t == 0 && L.pairs) atomicAdd(L.pairs, (unsigned long long)nr * (unsigned long long)S.ncols);
    if (warp >= 4) return;
    float dmax = 0.f;
    if (valid && ok) {
        const int r = r0 + t;
        if (!(tot >= 0x1p-60f && tot <= 0x1p60f)) {
            const int q = atomicAdd(L.n_fallback, 1);
            if (q < L.fallback_cap) L.fallback[q] = make_int4(item.x, r, blk, 0);
        } else {
            const double tilde = -(double)I.lam * L.eps_ln2 * ((double)Mi + log2((double)tot));
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

// Column tiles of one side: tile g of cluster J = tile_cl[g] holds columns off[J] + 128 (g - tile0[J]) + c,
// c < 128 (past the cluster's end: zero), centred at c_J and split; half_norm = |yh|^2 / 2.  Written into both
// copies (one per instance that uses the side as columns) at once; a null dst1 means one copy.
template <int NP, int K>
__global__ void __launch_bounds__(kN) tcc_build_kernel(const float *pts, int D4, const int *off, const int *tile0,
                                                       const int *tile_cl, const float *cen, unsigned char *dst0,
                                                       unsigned char *dst1, float *half_norm) {
    const int g = blockIdx.x, c = threadIdx.x;
    const int J = tile_cl[g];
    const int j = off[J] + (g - tile0[J]) * kN + c;
    const bool ok = j < off[J + 1];
    const size_t o = (size_t)g * xt::tile_bytes(NP, K);
    half_norm[(size_t)g * kN + c] = xt::build_col<NP, K, double>(pts + (size_t)(ok ? j : 0) * D4, cen + (size_t)J * D4, D4, ok, c,
                                                         dst0 + o, dst1 ? dst1 + o : nullptr);
}

// Per step: H_j = s (eps log w_j + pot_j - |yh_j|^2 / 2) into the column tiles of every instance (past a cluster's
// end, or for w_j = 0: a large negative H).
struct TccUpdate {
    unsigned char *tiles[kMaxInst];
    const float *half_norm[kMaxInst];
    const float *logw[kMaxInst];
    const float *pot[kMaxInst];
    const int *off[kMaxInst], *tile0[kMaxInst], *tile_cl[kMaxInst];
    int ntiles[kMaxInst];
    float s, eps;
};

template <int NP, int K> __global__ void tcc_update_kernel(const __grid_constant__ TccUpdate U) {
    const int q = blockIdx.y, c = threadIdx.x;
    for (int g = blockIdx.x; g < U.ntiles[q]; g += gridDim.x) {
        const int J = U.tile_cl[q][g];
        const int j = U.off[q][J] + (g - U.tile0[q][J]) * kN + c;
        double H = -1e30;  // in double: three terms that cancel, once per column and step
        if (j < U.off[q][J + 1])
            H = (double)U.s * ((double)U.eps * U.logw[q][j] + (double)U.pot[q][j] - U.half_norm[q][(size_t)g * kN + c]);
        xt::put_h<NP, K>(U.tiles[q] + (size_t)g * xt::tile_bytes(NP, K), c, (float)H, (float)(H - (double)(float)H));
    }
}

// f.template operator()<NP, K>() for the run-time pieces and slots
template <class F> void dispatch(int np, int K, F &&f) {
    switch (np * 100 + K) {
        case 232: f.template operator()<2, 32>(); break;
        case 248: f.template operator()<2, 48>(); break;
        case 264: f.template operator()<2, 64>(); break;
        case 316: f.template operator()<3, 16>(); break;
        case 332: f.template operator()<3, 32>(); break;
        case 348: f.template operator()<3, 48>(); break;
        case 364: f.template operator()<3, 64>(); break;
        default: throw Error{OTGB_EINTERNAL, "cluster-tiled form: unsupported pieces or width"};
    }
}

struct BuildFn {
    const float *pts;
    int D4;
    const int *off, *tile0, *tile_cl;
    int ntiles;
    const float *cen;
    unsigned char *dst0, *dst1;
    float *half_norm;
    cudaStream_t st;
    template <int NP, int K> void operator()() const {
        tcc_build_kernel<NP, K><<<ntiles, kN, 0, st>>>(pts, D4, off, tile0, tile_cl, cen, dst0, dst1, half_norm);
    }
};
struct UpdateFn {
    const TccUpdate &U;
    dim3 grid;
    cudaStream_t st;
    template <int NP, int K> void operator()() const { tcc_update_kernel<NP, K><<<grid, kN, 0, st>>>(U); }
};
struct SweepFn {
    const SoftminLaunch &L;
    int D4;
    cudaStream_t st;
    template <int NP, int K> void operator()() const {
        constexpr int bytes = xt::Geom<NP, K>::stages * xt::Geom<NP, K>::tile + (int)sizeof(TccCtl);
        static_assert(2 * (bytes + 1024) <= 227 * 1024, "two CTAs per SM");
        static PerDevice<int> attr;
        attr.get([] {
            OTGB_CUDA_TRY(cudaFuncSetAttribute(softmin_tcc_kernel<NP, K>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
            return 1;
        });
        softmin_tcc_kernel<NP, K><<<L.n_items, kThreads, bytes, st>>>(L, D4);
    }
};

}  // namespace

size_t tcc_tile_bytes(int np, int D4) { return (size_t)xt::tile_bytes(np, xt::k_slots(D4)); }

void tcc_build_side(int np, const float *pts, int D4, const int *d_off, const int *d_tile0, const int *d_tile_cl,
                    int ntiles, const float *cen, unsigned char *dst0, unsigned char *dst1, float *half_norm,
                    cudaStream_t st) {
    require(D4 <= 60, "tcc_build_side: D4 must be <= 60", OTGB_EINTERNAL);
    if (ntiles <= 0) return;
    dispatch(np, xt::k_slots(D4), BuildFn{pts, D4, d_off, d_tile0, d_tile_cl, ntiles, cen, dst0, dst1, half_norm, st});
    OTGB_CHECK_LAUNCH();
}

void tcc_update(const SoftminLaunch &L, int D, cudaStream_t st) {
    TccUpdate U;
    int mx = 0;
    for (int q = 0; q < kMaxInst; ++q) {
        const SoftminInst &I = L.inst[q];
        U.tiles[q] = const_cast<unsigned char *>(I.tcc_tiles);
        U.half_norm[q] = I.tcc_half_norm;
        U.logw[q] = I.col_logw;
        U.pot[q] = I.col_pot;
        U.off[q] = I.tcc_coff;
        U.tile0[q] = I.tcc_tile0;
        U.tile_cl[q] = I.tcc_tile_cl;
        U.ntiles[q] = q < L.n_inst ? I.tcc_ntiles : 0;
        mx = std::max(mx, U.ntiles[q]);
    }
    U.s = L.s;
    U.eps = L.eps;
    if (mx <= 0) return;
    dispatch(L.use_tcc, xt::k_slots((D + 3) & ~3), UpdateFn{U, dim3(std::min(mx, 65535), L.n_inst), st});
    OTGB_CHECK_LAUNCH();
}

void softmin_tcc_launch(const SoftminLaunch &L, int D, cudaStream_t st) {
    const int D4 = (D + 3) & ~3;
    require(D4 <= 60 && L.tcc_nwords <= kMaxWords, "softmin_tcc_launch: unsupported shape", OTGB_EINTERNAL);
    dispatch(L.use_tcc, xt::k_slots(D4), SweepFn{L, D4, st});
    OTGB_CHECK_LAUNCH();
}

}  // namespace otgb
