// FP64 n2 pass on the line engine, line lengths of list A.
#include "hom_passes.cuh"

namespace hom {
F64X2Fn f64_x2_kernel_a(int n, int inverse) {
    switch (n) {
#define HOM_CASE(N) case N: return inverse ? k_x2<double, 1, N> : k_x2<double, -1, N>;
        HOM_F64_LENGTHS_A(HOM_CASE)
#undef HOM_CASE
        default: return nullptr;
    }
}
}  // namespace hom
