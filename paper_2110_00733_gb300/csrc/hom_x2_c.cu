// TMA-staged n2 pass (FP32), line lengths of list C.
#include "hom_lines.cuh"

namespace hom {
X2LineFn x2_line_kernel_c(int n, int inverse) {
    switch (n) {
#define HOM_CASE(N) case N: return inverse ? k_x2_tma<float, 1, N> : k_x2_tma<float, -1, N>;
        HOM_LINE_LENGTHS_C(HOM_CASE)
#undef HOM_CASE
        default: return nullptr;
    }
}
}  // namespace hom
