// FP64 n3 pass on the line engine, line lengths of list B.
#include "hom_passes.cuh"

namespace hom {
F64X3Fn f64_x3_kernel_b(int n, int pairs) {
    switch (n) {
#define HOM_CASE(N) case N: return pairs == 5 ? k_x3<double, N, 5> : k_x3<double, N, 3>;
        HOM_LINE_LENGTHS_B(HOM_CASE)
#undef HOM_CASE
        default: return nullptr;
    }
}
}  // namespace hom
