// Fused MINRES n1 pass (FP32), line lengths of list B.
#include "hom_lines.cuh"

namespace hom {
X1lLineFn x1l_line_kernel_b(int n) {
    switch (n) {
#define HOM_CASE(N) case N: if constexpr (x1l_cols(N, LinePlan<N>::TPL) > 0) return k_x1_lanczos_tma<float, N>; else return nullptr;
        HOM_LINE_LENGTHS_B(HOM_CASE)
#undef HOM_CASE
        default: return nullptr;
    }
}
}  // namespace hom
