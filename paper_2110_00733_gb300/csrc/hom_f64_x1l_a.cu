// FP64 fused MINRES n1 pass on the line engine, line lengths of list A.
#include "hom_passes.cuh"

namespace hom {
F64X1lFn f64_x1l_kernel_a(int n) {
    switch (n) {
#define HOM_CASE(N) case N: return k_x1_lanczos<double, N>;
        HOM_F64_LENGTHS_A(HOM_CASE)
#undef HOM_CASE
        default: return nullptr;
    }
}
}  // namespace hom
