// Large dense D <= 3 sums over spatially sorted points (sorted3.cu).
#pragma once

#include "otgb_internal.cuh"

namespace otgb {

// One sum of the gradient: columns (x, y, z, log w) with a potential, against the rows' potential.
struct Grad3Part {
    const float4 *cols;
    const float *pot;
    int n;
    float sign;
    const float *row_pot;
};
// grad[perm[r]] (+)= row_w[r] scale sum_parts sign sum_j w_j exp((row_pot_r + pot_j - |x_r - y_j|^2 / 2) / eps) (x_r - y_j)
// over every pair; rows and columns in an order in which neighbours in the order are neighbours in space.
void grad3_run(otgb_ctx *ctx, const float4 *rows, int n, int D, const Grad3Part (&part)[2], double eps, const float *row_w,
               float scale, int accumulate, const int *perm, float *grad, cudaStream_t st);

// sinkhorn_grad_x for D <= 3, p = 2 from the caller's arrays (sorts, then grad3_run).
void grad3_apply(otgb_ctx *ctx, const float *x, const float *alpha, int N, const float *y, const float *beta, int M, int D,
                 double eps, const float *f, const float *g, const float *a_self, float *grad);

// otgb_softmin for D <= 3: sorts rows and columns and visits the column tiles that can matter.
void softmin3_sorted(otgb_ctx *ctx, const float *q, int n_out, const float *p, const float *w, const float *pot, int n_in,
                     int D, double eps, double lam, const float *old, double omega, float *out, const float *d_box,
                     const float *d_cen);

}  // namespace otgb
