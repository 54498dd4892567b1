// hom_sum3.h -- a sum of products of floats held as three floats.  Plain C++, so
// that it can be run on the host (-ffp-contract=off there: every operation rounds
// by itself).
#pragma once
#include <math.h>

#ifdef __CUDACC__
#define HOM_SUM_HD __host__ __device__ __forceinline__
#else
#define HOM_SUM_HD inline
#endif

namespace hom {

#ifdef __CUDA_ARCH__
HOM_SUM_HD float rn_add(float a, float b) { return __fadd_rn(a, b); }
HOM_SUM_HD float rn_mul(float a, float b) { return __fmul_rn(a, b); }
HOM_SUM_HD float rn_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
#else
HOM_SUM_HD float rn_add(float a, float b) { return a + b; }
HOM_SUM_HD float rn_mul(float a, float b) { return a * b; }
HOM_SUM_HD float rn_fma(float a, float b, float c) { return fmaf(a, b, c); }
#endif

// s + b -> (s, its rounding error), Knuth's two-sum
HOM_SUM_HD float two_sum(float &s, float b) {
    const float a = s;
    s = rn_add(a, b);
    const float bb = rn_add(s, -a);
    return rn_add(rn_add(a, -rn_add(s, -bb)), rn_add(b, -bb));
}

// Each product exactly as two floats, the leading parts and then what their sum and
// the products' tails leave each added with their errors kept; only the third float
// rounds, below 2^-70 of the sum.  Two floats are not enough where FP64 stood: they
// drop the tails' last bits, and squares have those mostly set (an odd square is 1
// mod 8), so that a sum of squares comes out 8e-16 small whatever the number of
// threads it is spread over (FP64: 1e-16).
struct Sum3 {
    float hi = 0.f, lo = 0.f, low = 0.f;
    HOM_SUM_HD void add_prod(float a, float b) {
        const float p = rn_mul(a, b), e = rn_fma(a, b, -p);
        const float r = two_sum(hi, p);
        const float r1 = two_sum(lo, r), r2 = two_sum(lo, e);
        low = rn_add(low, rn_add(r1, r2));
    }
    HOM_SUM_HD double value() const { return (double)hi + ((double)lo + (double)low); }
};

}  // namespace hom
