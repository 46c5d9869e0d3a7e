// Dense softmin sweep for 3 < D, D4 <= 60 at float32 accuracy on the tensor cores: three-piece BF16 operands
// (xtile.cuh), the pair centred at the row block's mean as in softmin_gen_kernel, every block against a range of
// consecutive columns.
//
//   MAXP = false: the shift of a row comes from its old value (M_i = -s old_i / lam) and rides in the row operand.
//   MAXP = true:  no old value (otgb_softmin, the extrapolation): each thread keeps a running shift of its row.  The
//     accumulator holds the pair's whole base-2 exponent, so one pass does: 32 exponents at a time, their maximum,
//     the running sum rescaled when the maximum passes the shift by 30 binades (a sum stays below 2^30 n), then ex2.
//     softmin_gen_kernel swept the columns twice instead (maximum, then sum).
//
// One CTA: warps 0-3 one row per thread (row operand into tensor memory, sums), warps 4-7 one column per thread
// (centre, split, store a tile's column operand), warp 8 one lane: bulk copies of the raw columns, two tiles ahead,
// and the MMAs.  Two CTAs share an SM (about 111 KB of shared memory, 256 tensor-memory columns each): a CTA's tile
// period is build (about 600 clocks) + MMA (1536 at K = 64), so that two CTAs keep the tensor pipe busy although each
// holds one column operand and one accumulator.
//
// Bound: the tensor pipe, six products, 2.49e12 pairs/s at K = 64 (4e8 pairs: 0.16 ms).  Measured, otgb_softmin of
// 20k x 20k fibers (60-D): 5.42 -> 0.375 ms for the whole call, 0.32 of it this kernel (softmin_gen_kernel: two sweeps,
// 157 CTAs for 304 slots); error against FP64 (rms, of the largest result) 1.3e-6 -> 0.7e-6.  Extrapolation at 300k per side: 4.5 -> 2.3 ms.
//
// Columns of a block may be split over several items (SoftminLaunch::part: shift and sum per row, combined in item
// order by the CTA that completes the block's last item).
#include <cfloat>
#include <cmath>

#include "otgb_internal.cuh"
#include "xtile.cuh"

namespace otgb {
namespace {

constexpr int kThreads = 288;
constexpr int kN = xt::kCols;
constexpr float kNoTerm = -1e29f;  // shift of a row without terms (absent columns have an exponent of about -1e30)

template <int K> struct XdSmem {
    static constexpr int kW = K - 4;  // widest point
    alignas(1024) unsigned char b[xt::tile_bytes(3, K)];
    alignas(16) float raw[2][kN * kW];
    float cen[kW];
    float csum[4][kW];
    unsigned long long raw_full[2], b_full, b_empty, acc_full, acc_free, a_ready, drain;
    float tmax[4];  // largest T of the rows, per warp
    uint32_t tslot;
    int abort;
    int bc[2];
};

template <int K, bool MAXP>
__global__ void __launch_bounds__(kThreads, 2) softmin_xd_kernel(const __grid_constant__ SoftminLaunch L, int D4) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    XdSmem<K> &S = *reinterpret_cast<XdSmem<K> *>(smem_raw);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    int4 item = L.items[blockIdx.x];
    OTGB_DCLAMP(item.x, 0, L.n_inst);
    const SoftminInst &I = L.inst[item.x];
    const int blk = item.y;
    int r0 = I.blk_row0[blk], r1 = I.blk_row0[blk + 1];
    OTGB_DCLAMP(r0, 0, I.n_rows + 1);
    OTGB_DCLAMP(r1, r0, min(I.n_rows, r0 + xt::kRows) + 1);
    const int nr = r1 - r0;
    int cb = item.z, ce = item.w;
    OTGB_DCLAMP(cb, 0, I.n_cols + 1);
    OTGB_DCLAMP(ce, cb, I.n_cols + 1);
    const int ncol = ce - cb, ntiles = (ncol + kN - 1) / kN;
    const float s = L.s;
    volatile int *abort = &S.abort;

    if (t == 0) {
        S.abort = 0;
        tc::mbar_init(&S.raw_full[0], 1);
        tc::mbar_init(&S.raw_full[1], 1);
        tc::mbar_init(&S.b_full, 128);
        tc::mbar_init(&S.b_empty, 1);
        tc::mbar_init(&S.acc_full, 1);
        tc::mbar_init(&S.acc_free, 128);
        tc::mbar_init(&S.a_ready, 128);
        tc::mbar_init(&S.drain, 1);
        tc::mbar_init_fence();
    }
    if (warp == 8) tc::tmem_alloc(&S.tslot, xt::kTmemCols);
    // centre: the mean of the block's rows (thread t: coordinate t % 64 over every fourth row)
    if (t < 256 && (t & 63) < D4) {
        const float *p = I.rows + (size_t)r0 * D4 + (t & 63);
        float acc = 0.f;
        for (int r = t >> 6; r < nr; r += 4) acc += p[(size_t)r * D4];
        S.csum[t >> 6][t & 63] = acc;
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (t < D4) S.cen[t] = nr > 0 ? ((S.csum[0][t] + S.csum[1][t]) + (S.csum[2][t] + S.csum[3][t])) / (float)nr : 0.f;
    const uint32_t tmem = S.tslot;
    __syncthreads();

    float tot = 0.f, sh = kNoTerm, Mi = 0.f;
    bool far_row = false;
    if (warp == 8) {
        if (lane == 0) {
            bool ok = true;
            auto copy = [&](int k) {
                const int n = min(kN, ncol - k * kN);
                xt::tma_load(S.raw[k & 1], I.cols + (size_t)(cb + k * kN) * D4, (uint32_t)(n * D4 * 4), &S.raw_full[k & 1]);
            };
            int copied = 0;
            for (; copied < 2 && copied < ntiles; ++copied) copy(copied);
            if (ntiles > 0) ok = xt::wait(&S.a_ready, 0, abort);
            const bool last = !MAXP && xt::fold_last(S.tmax);  // without old values the rows come as they are
            for (int k = 0; ok && k < ntiles; ++k) {
                ok = xt::wait(&S.b_full, (uint32_t)(k & 1), abort);
                if (!ok) break;
                // the builders are done with the raw columns of tile k
                if (copied < ntiles) copy(copied++);
                ok = k == 0 || xt::wait(&S.acc_free, (uint32_t)((k - 1) & 1), abort);
                if (!ok) break;
                tc::fence_after();
                xt::issue<3, K>(tmem, tmem + kN, tc::smem_u32(S.b), last ? xt::kFoldLast : k & 1);
                tc::commit(&S.b_empty);
                tc::commit(&S.acc_full);
            }
            // nothing in flight at exit: every MMA completed, the last copy into each buffer landed
            tc::commit(&S.drain);
            if (!tc::mbar_wait(&S.drain, 0)) ok = false;
            for (int q = max(0, copied - 2); q < copied; ++q)
                if (!tc::mbar_wait(&S.raw_full[q & 1], (uint32_t)((q >> 1) & 1))) ok = false;
            if (!ok) *abort = 1;
        }
        __syncwarp();
    } else if (warp >= 4) {
        // ------------------------------------------------------- column operands
        const int c = t - 128;
        bool ok = true;
        // log weight and potential of this thread's column, one tile ahead
        auto fetch = [&](int k, float &lw, float &pot) {
            const int j = k * kN + c;
            lw = -INFINITY;
            pot = 0.f;
            if (j < ncol) {
                lw = I.col_logw[cb + j];
                pot = I.col_pot[cb + j];
            }
        };
        float lw, pot;
        if (ntiles > 0) fetch(0, lw, pot);
        for (int k = 0; k < ntiles; ++k) {
            ok = xt::wait(&S.raw_full[k & 1], (uint32_t)((k >> 1) & 1), abort);
            if (ok && k > 0) ok = xt::wait(&S.b_empty, (uint32_t)((k - 1) & 1), abort);
            if (!ok) {
                *abort = 1;
                break;
            }
            const bool in = k * kN + c < ncol;
            const float hn = xt::build_col<3, K, float>(S.raw[k & 1] + c * D4, S.cen, D4, in, c, S.b, nullptr);
            xt::put_h_sum<3, K>(S.b, c, s, L.eps, lw, pot, hn);
            tc::fence_proxy_async();
            xt::arrive(&S.b_full);
            if (k + 1 < ntiles) fetch(k + 1, lw, pot);
        }
    } else {
        // --------------------------------------------------- row operand and sums
        const uint32_t lanes = tmem + ((uint32_t)(warp * 32) << 16);
        const bool valid = t < nr;
        {
            float x[K - 4];
            const float4 *x4 = reinterpret_cast<const float4 *>(I.rows + (size_t)(r0 + (valid ? t : 0)) * D4);
#pragma unroll
            for (int q = 0; q < K / 4 - 1; ++q) {
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (valid && 4 * q < D4) v = x4[q];
                x[4 * q] = v.x;
                x[4 * q + 1] = v.y;
                x[4 * q + 2] = v.z;
                x[4 * q + 3] = v.w;
            }
            if (!MAXP && valid) Mi = (float)(-(double)s * (double)I.row_old[r0 + t] / (double)I.lam);
            const float T = xt::stage_row<3, K>(x, D4, S.cen, s, Mi, valid, lanes + kN);
            if constexpr (!MAXP) xt::put_t(T, &S.tmax[warp], lane);
            else far_row = T > xt::kFarRow;
        }
        xt::st_wait();
        tc::fence_before();
        xt::arrive(&S.a_ready);
        for (int k = 0; k < ntiles; ++k) {
            if (!__all_sync(0xffffffffu, xt::wait(&S.acc_full, (uint32_t)(k & 1), abort))) {
                *abort = 1;  // tensor-memory loads are warp-collective
                break;
            }
            tc::fence_after();
            auto freed = [&] {
                tc::fence_before();
                xt::arrive(&S.acc_free);
            };
            if constexpr (MAXP) xt::sum_row_max(lanes, tot, sh, freed);
            else tot = xt::sum_row(lanes, tot, freed);
        }
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const bool ok = S.abort == 0;
    if (!ok && t == 0 && L.tc_err) atomicOr(L.tc_err, 1u);
    if (warp == 8) tc::tmem_dealloc(tmem, xt::kTmemCols);
    if (t == 0 && L.pairs) atomicAdd(L.pairs, (unsigned long long)nr * (unsigned long long)ncol);
    if (!ok) return;  // uniform
    if (L.part) {
        // split block: (shift, sum) per row; the CTA that completes the block's last item combines them in item order
        float2 *part = reinterpret_cast<float2 *>(L.part);
        if (t < xt::kRows) part[(size_t)blockIdx.x * kPartRows + t] = make_float2(sh, tot);
        __threadfence();
        __syncthreads();
        if (t == 0) {
            int fi = L.item_fin[blockIdx.x];
            OTGB_DCLAMP(fi, 0, L.n_fin);
            S.bc[0] = fi;
            S.bc[1] = atomicAdd(L.fin_count + fi, 1) + 1;
        }
        __syncthreads();
        const int4 fe = L.fin[S.bc[0]];
        if (S.bc[1] != fe.w) return;  // uniform
        __threadfence();
        if (t < xt::kRows) {
            const float2 *p = part + (size_t)fe.z * kPartRows + t;
            sh = kNoTerm;
            for (int q = 0; MAXP && q < fe.w; ++q) sh = fmaxf(sh, __ldcg(&p[(size_t)q * kPartRows]).x);
            tot = 0.f;
            for (int q = 0; q < fe.w; ++q) {
                const float2 v = __ldcg(&p[(size_t)q * kPartRows]);
                tot += MAXP ? v.y * xt::ex2(v.x - sh) : v.y;
            }
        }
    }
    if (warp >= 4) return;
    float dmax = 0.f;
    if (t < nr) {
        const int r = r0 + t;
        if (!(tot >= 0x1p-60f && tot <= 0x1p60f) || far_row) {
            const int q = atomicAdd(L.n_fallback, 1);
            if (q < L.fallback_cap) L.fallback[q] = make_int4(item.x, r, blk, 0);
        } else {
            const double L2 = (MAXP ? (double)sh : (double)Mi) + log2((double)tot);
            const double tilde = -(double)I.lam * L.eps_ln2 * L2;
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

template <int K, bool MAXP> void launch(const SoftminLaunch &L, int D4, cudaStream_t st) {
    static_assert(2 * (sizeof(XdSmem<K>) + 1024) <= 228 * 1024, "two CTAs per SM");
    static PerDevice<int> attr;
    attr.get([] {
        OTGB_CUDA_TRY(cudaFuncSetAttribute(softmin_xd_kernel<K, MAXP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)sizeof(XdSmem<K>)));
        return 1;
    });
    softmin_xd_kernel<K, MAXP><<<L.n_items, kThreads, sizeof(XdSmem<K>), st>>>(L, D4);
}

}  // namespace

void softmin_xd_launch(const SoftminLaunch &L, int D, bool maxp, cudaStream_t st) {
    const int D4 = (D + 3) & ~3;
    switch (xt::k_slots(D4) + (maxp ? 1 : 0)) {
        case 16: launch<16, false>(L, D4, st); break;
        case 17: launch<16, true>(L, D4, st); break;
        case 32: launch<32, false>(L, D4, st); break;
        case 33: launch<32, true>(L, D4, st); break;
        case 48: launch<48, false>(L, D4, st); break;
        case 49: launch<48, true>(L, D4, st); break;
        case 64: launch<64, false>(L, D4, st); break;
        case 65: launch<64, true>(L, D4, st); break;
        default: throw Error{OTGB_EINTERNAL, "softmin_xd_launch: unsupported width"};
    }
    OTGB_CHECK_LAUNCH();
}

int split_chunk(const std::vector<std::pair<long long, long long>> &blocks_cols, long long slots) {
    // The split into chunks of c tiles that minimises waves x (c + 3), the set-up of an item (tensor memory, centre, row
    // operand, first copies: 3 to 4 us) counted as three tiles.
    long long tmax = 1;
    for (auto &bc : blocks_cols) tmax = std::max(tmax, (bc.second + kN - 1) / kN);
    long long best = tmax, cost = -1;
    for (long long parts = 1; parts <= tmax; ++parts) {
        const long long c = (tmax + parts - 1) / parts;
        long long items = 0;
        for (auto &bc : blocks_cols) items += bc.first * (((bc.second + kN - 1) / kN + c - 1) / c);
        const long long v = (items + slots - 1) / slots * (c + 3);
        if (cost < 0 || v < cost) {
            cost = v;
            best = c;
        }
        if (items > 16 * slots) break;
    }
    return (int)std::min<long long>(best * kN, 1 << 30);
}

}  // namespace otgb
