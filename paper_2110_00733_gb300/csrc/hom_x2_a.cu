// TMA-staged n2 pass (FP32), line lengths of list A.
#include "hom_lines.cuh"

namespace hom {
X2LineFn x2_line_kernel_a(int n, int inverse) {
    switch (n) {
#define HOM_CASE(N) case N: return inverse ? k_x2_tma<float, 1, N> : k_x2_tma<float, -1, N>;
        HOM_LINE_LENGTHS_A(HOM_CASE)
#undef HOM_CASE
        default: return nullptr;
    }
}
}  // namespace hom
