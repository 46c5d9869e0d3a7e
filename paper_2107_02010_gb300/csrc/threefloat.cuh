// A sum in three floats (some 70 bits: Knuth's two-sum, Dekker's product by FMA), for sums that are held in FP64 elsewhere.  The
// FP64 units of this GPU do two operations per clock and SM, so that double sums over the coordinates of all points bounded
// their kernel; a step here is some twenty FP32 operations, and rounds less than a double sum does.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define OTGB_HD __host__ __device__ __forceinline__
#else
#define OTGB_HD inline
#endif

namespace otgb {

struct ThreeFloat {
    float hi = 0.f, mid = 0.f, lo = 0.f;
    bool exact = true;  // false: a product came so near the denormal range that its error term may be lost

    static OTGB_HD float add_(float a, float b) {
#ifdef __CUDA_ARCH__
        return __fadd_rn(a, b);  // never part of an FMA
#else
        return a + b;
#endif
    }
    // a + b = s + e
    static OTGB_HD void two_sum(float a, float b, float &s, float &e) {
        s = add_(a, b);
        const float bb = add_(s, -a);
        e = add_(add_(a, -add_(s, -bb)), add_(b, -bb));
    }
    OTGB_HD void add_small(float v) {
        float e;
        two_sum(mid, v, mid, e);
        lo = add_(lo, e);
    }
    OTGB_HD void add(float v) {
        float e;
        two_sum(hi, v, hi, e);
        add_small(e);
    }
    OTGB_HD void add_product(float a, float b) {
#ifdef __CUDA_ARCH__
        const float p = __fmul_rn(a, b);
#else
        const float p = a * b;
#endif
        exact = exact && (fabsf(p) >= 0x1p-100f || a == 0.f || b == 0.f);
        add(p);
        add_small(fmaf(a, b, -p));
    }
    OTGB_HD bool usable() const { return exact && fabsf(hi) <= 3.4e38f && fabsf(mid) <= 3.4e38f; }  // no NaN, no infinity
    OTGB_HD double value() const { return (double)hi + ((double)mid + (double)lo); }
};

}  // namespace otgb
