// Label transfer on the tensor cores (transport_xt.cu), called by transport_apply (transport.cu).
#pragma once

#include "otgb_internal.cuh"

namespace otgb {

struct TransportCall {
    const float *x, *y, *b;  // caller layout
    int N, M, D, L;
    double eps;
    const float *f, *g;      // caller order
    const int *labels;
    const float *d_cen;      // common centre (64 floats)
    float *scores;           // caller's outputs; scores and row_mass may be null
    int *argmax;
    float *row_mass;
};
// What the safe kernel needs for the rows listed in fallback: packed rows and sorted columns, the rows' caller order.
struct TransportFallback {
    const float *rows, *f, *cols, *col_logw, *g;
    const int *col_lab, *row_perm;
    int4 *fallback;
    int *n_fallback;
};
// Columns by label (stable; labels outside [0, L) last): sorted keys, order, first position of each class (L + 1).
void label_order(otgb_ctx *ctx, const int *labels, int M, int L, uint32_t *keys, int *perm, int *lab_off);
// Near ties in numbers: transport_gen_kernel over the blocks that hold one, the classes marked in cls_bits (per block), writing
// the argmax of the rows marked in tied.  rows, f: in the order perm of that kernel; cols, col_logw, g: sorted by label.
struct TieBlocks {
    const float *rows, *f, *cols, *col_logw, *g;
    const int *blk_row0, *lab_off, *perm;
    int nblk, n, m, D, L;
    float eps, s;
    const unsigned *cls_bits;
    const unsigned char *tied;
    int *argmax;
};
void transport_gen_ties(const TieBlocks &T, cudaStream_t st);
// 3 < D, D4 <= 60.
TransportFallback transport_xt_apply(otgb_ctx *ctx, const TransportCall &c);

}  // namespace otgb
