// FP64-field instantiation of the FFT passes and Krylov kernels.
#include "hom_passes.cuh"

namespace hom {
template struct Launch<double>;

F64X1Fn f64_x1_kernel_a(int n), f64_x1_kernel_b(int n), f64_x1_kernel_c(int n);
F64X1Fn f64_x1_kernel(int n) {
    F64X1Fn f = f64_x1_kernel_a(n);
    if (!f) f = f64_x1_kernel_b(n);
    return f ? f : f64_x1_kernel_c(n);
}

F64X1lFn f64_x1l_kernel_a(int n), f64_x1l_kernel_b(int n), f64_x1l_kernel_c(int n);
F64X1lFn f64_x1l_kernel(int n) {
    F64X1lFn f = f64_x1l_kernel_a(n);
    if (!f) f = f64_x1l_kernel_b(n);
    return f ? f : f64_x1l_kernel_c(n);
}

F64X2Fn f64_x2_kernel_a(int n, int inverse), f64_x2_kernel_b(int n, int inverse), f64_x2_kernel_c(int n, int inverse);
F64X2Fn f64_x2_kernel(int n, int inverse) {
    F64X2Fn f = f64_x2_kernel_a(n, inverse);
    if (!f) f = f64_x2_kernel_b(n, inverse);
    return f ? f : f64_x2_kernel_c(n, inverse);
}

F64X3Fn f64_x3_kernel_a(int n, int pairs), f64_x3_kernel_b(int n, int pairs), f64_x3_kernel_c(int n, int pairs);
F64X3Fn f64_x3_kernel(int n, int pairs) {
    F64X3Fn f = f64_x3_kernel_a(n, pairs);
    if (!f) f = f64_x3_kernel_b(n, pairs);
    return f ? f : f64_x3_kernel_c(n, pairs);
}
F64X1Fn f64_ord_x1_kernel_a(int n), f64_ord_x1_kernel_b(int n);
F64X1Fn f64_ord_x1_kernel(int n) {
    F64X1Fn f = f64_ord_x1_kernel_a(n);
    return f ? f : f64_ord_x1_kernel_b(n);
}

F64X2Fn f64_ord_x2_kernel_a(int n, int inverse), f64_ord_x2_kernel_b(int n, int inverse);
F64X2Fn f64_ord_x2_kernel(int n, int inverse) {
    F64X2Fn f = f64_ord_x2_kernel_a(n, inverse);
    return f ? f : f64_ord_x2_kernel_b(n, inverse);
}

F64X3Fn f64_ord_x3_kernel_a(int n), f64_ord_x3_kernel_b(int n);
F64X3Fn f64_ord_x3_kernel(int n) {
    F64X3Fn f = f64_ord_x3_kernel_a(n);
    return f ? f : f64_ord_x3_kernel_b(n);
}
}
