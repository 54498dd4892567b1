// FP64 n1 pass on the line engine, line lengths of list A.
#include "hom_passes.cuh"

namespace hom {
F64X1Fn f64_x1_kernel_a(int n) {
    switch (n) {
#define HOM_CASE(N) case N: return k_x1<double, N>;
        HOM_F64_LENGTHS_A(HOM_CASE)
#undef HOM_CASE
        default: return nullptr;
    }
}
}  // namespace hom
