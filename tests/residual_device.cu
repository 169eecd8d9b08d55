// C entry point to the tensor-core GEMM with its residual |I - C|^2 (csrc/k_tc.cu), for the GPU tests.  Test
// infrastructure: built by tests/test_gpu_tc_residual.py and linked to the library.
#include "internal.h"

using namespace mbdgb;

// C = A B^T (TF32x3 parts, order n), resid += |I - C|^2 over the leading nvalid rows and columns.
extern "C" int tc_residual(const float *A0, const float *A1, const float *B0, const float *B1, float *C, int n, int nvalid,
                           double *resid, int *err) {
    const TcOperands op{A0, A1, B0, B1, n, n};
    const TcArgs g{n, n, n, 1.f, 0.f, nullptr, n, C, nullptr, nullptr, nullptr, nullptr, nullptr, resid, nvalid, 0, err};
    return static_cast<int>(tc_gemm(2, op, g, nullptr));
}
