// FP64 n1 pass on the line engine, line lengths of list B.
#include "hom_passes.cuh"

namespace hom {
F64X1Fn f64_x1_kernel_b(int n) {
    switch (n) {
#define HOM_CASE(N) case N: return k_x1<double, N>;
        HOM_LINE_LENGTHS_B(HOM_CASE)
#undef HOM_CASE
        default: return nullptr;
    }
}
}  // namespace hom
