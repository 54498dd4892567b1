// Persistent n3 pass (FP32), lengths of list C.
#include "hom_x3.cuh"

namespace hom {
X3Line x3_line_kernel_c(int n) {
    switch (n) {
#define HOM_CASE(N) case N: return X3Line{k_x3_line<N, false>, k_x3_line<N, true>, X3Plan<N>::NT, X3Plan<N>::ROWS, X3Plan<N>::SMEM};
        HOM_X3_LENGTHS_C(HOM_CASE)
#undef HOM_CASE
        default: return X3Line{};
    }
}
}  // namespace hom
