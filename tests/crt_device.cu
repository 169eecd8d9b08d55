// C entry points to the residue products of the CUDA library (csrc/k_crt.cu) on device pointers,
// for the GPU tests.  Test infrastructure: built by tests/test_gpu_crt.py and linked to the library.
#include "internal.h"

using namespace mbdgb;

extern "C" size_t crt_real_bytes(int M, int N, int K) { return crt_gemm_bytes(M, N, K); }
extern "C" int crt_real(const double *A, long long lda, const double *Bt, long long ldb, int M, int N, int K, double alpha,
                        double beta, const double *D, long long ldd, double *C, long long ldc, double *T, long long ldt,
                        int sym, void *work, int *err) {
    CrtResult r{alpha, beta, D, C, T, ldd, ldc, ldt, 0, 0, 0, 0, 0, sym};
    return static_cast<int>(crt_gemm(A, lda, Bt, ldb, M, N, K, r, work, err, nullptr));
}

// Planar complex matrices of order n (pitch ld, planes and items as in the library): C = alpha A B + beta D.
extern "C" size_t crt_complex_bytes(int n, int batch) {
    return crt_operand_bytes(crt_shape(n, n, batch, true, false)) + crt_operand_bytes(crt_shape(n, n, batch, true, true)) +
           crt_bytes_bytes(n, crt_shape(n, n, batch, true, true).out_rows, batch);
}
extern "C" int crt_complex(const double *A, const double *B, int conj, int n, long long ld, int batch, double alpha,
                           double beta, const double *D, double *C, double *T, int sym, void *work, int *err) {
    const long long m2 = ld * ld;
    char *p = static_cast<char *>(work);
    const CrtShape sa = crt_shape(n, n, batch, true, false), sb = crt_shape(n, n, batch, true, true);
    const CrtOperand a = crt_rows(sa, A, A + m2, ld, 2 * m2, false, p, nullptr);
    p += crt_operand_bytes(sa);
    const CrtOperand b = crt_rows(sb, B, B + m2, ld, 2 * m2, conj != 0, p, nullptr);
    p += crt_operand_bytes(sb);
    CrtResult r{alpha, beta, D, C, T, ld, ld, ld, 2 * m2, 2 * m2, 2 * m2, m2, 0, sym};
    return static_cast<int>(crt_multiply(a, b, r, p, err, nullptr));
}

extern "C" size_t crt_cholesky_bytes(long long ld, int batch) { return cholesky_crt_bytes(ld, batch); }
extern "C" int crt_cholesky(double *A, long long ld, int batch, double *dinv, void *work, int *status) {
    return static_cast<int>(cholesky_crt(A, ld, ld * ld, batch, dinv, work, status, nullptr));
}
