// FP64 passes of the elastoplastic increments (ordered_fft), line lengths of list B.
#include "hom_passes.cuh"

namespace hom {
#define HOM_CASE(N, K)                                        \
    case N:                                                   \
        if constexpr (!is_fast_length(N)) return K;           \
        else return nullptr;
F64X1Fn f64_ord_x1_kernel_b(int n) {
    switch (n) {
#define HOM_CASE1(N) HOM_CASE(N, (k_x1<double, -N>))
        HOM_LINE_LENGTHS_B(HOM_CASE1)
        default: return nullptr;
    }
}
F64X2Fn f64_ord_x2_kernel_b(int n, int inverse) {
    switch (n) {
#define HOM_CASE2(N) HOM_CASE(N, (inverse ? k_x2<double, 1, -N> : k_x2<double, -1, -N>))
        HOM_LINE_LENGTHS_B(HOM_CASE2)
        default: return nullptr;
    }
}
F64X3Fn f64_ord_x3_kernel_b(int n) {
    switch (n) {
#define HOM_CASE3(N) HOM_CASE(N, (k_x3<double, -N, 3>))
        HOM_LINE_LENGTHS_B(HOM_CASE3)
        default: return nullptr;
    }
}
}  // namespace hom
