// FP32-field instantiation of the FFT passes and Krylov kernels.
#include "hom_passes.cuh"

namespace hom {
template struct Launch<float>;

X1lLineFn x1l_line_kernel_a(int n), x1l_line_kernel_b(int n), x1l_line_kernel_c(int n);
X1lLineFn x1l_line_kernel(int n) {
    X1lLineFn f = x1l_line_kernel_a(n);
    if (!f) f = x1l_line_kernel_b(n);
    return f ? f : x1l_line_kernel_c(n);
}

X3Line x3_line_kernel_a(int n), x3_line_kernel_b(int n), x3_line_kernel_c(int n);
X3Line x3_line_kernel(int n) {
    X3Line f = x3_line_kernel_a(n);
    if (!f.fn) f = x3_line_kernel_b(n);
    return f.fn ? f : x3_line_kernel_c(n);
}

X2LineFn x2_line_kernel_a(int n, int inverse), x2_line_kernel_b(int n, int inverse), x2_line_kernel_c(int n, int inverse);
X2LineFn x2_line_kernel(int n, int inverse) {
    X2LineFn f = x2_line_kernel_a(n, inverse);
    if (!f) f = x2_line_kernel_b(n, inverse);
    return f ? f : x2_line_kernel_c(n, inverse);
}
}
