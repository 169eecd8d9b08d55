// Host run of the residue arithmetic of the FP64 products (csrc/crt64.cuh: the functions the
// kernels of k_crt.cu call), for the CPU tests.  Test infrastructure: built by
// tests/test_crt_host.py into tests/_build.
#include "crt64.cuh"

using namespace mbdgb;

extern "C" int crt_moduli(int *m) {
    for (int i = 0; i < crt::kMod; ++i) m[i] = crt::kModuli[i];
    return crt::kMod;
}
extern "C" int crt_chunk() { return crt::kChunk * crt::kStageK; }
extern "C" int crt_exponent(double norm) { return crt::row_exponent(norm); }

// Residues [kMod][n] of the integers x [n], as k_crt_rows forms them.
extern "C" void crt_residues(const long long *x, int n, float *r) {
    for (int j = 0; j < n; ++j) {
        const crt::Limbs l = crt::limbs(x[j]);
        crt::each_modulus([&](auto I) { r[decltype(I)::value * n + j] = crt::residue<decltype(I)::value>(l); });
    }
}

// An accumulation's sum v mod m_i, as k_crt_gemm reduces it.
extern "C" void crt_reduce(int i, const float *v, int n, float *out) {
    const float m = static_cast<float>(crt::kModuli[i]), inv = 1.0f / m;
    for (int j = 0; j < n; ++j) out[j] = crt::reduce(v[j], m, inv);
}

// The stored byte of a residue, and the result from the bytes y [kMod][n]: x.y / P 2^64.
extern "C" void crt_stored(int i, const float *r, int n, float *y) {
    const float m = static_cast<float>(crt::kModuli[i]), inv = 1.0f / m;
    for (int j = 0; j < n; ++j) y[j] = crt::stored(r[j], m, inv, static_cast<float>(crt::inverse_of_rest(i)));
}
extern "C" double crt_result(const unsigned char *y, int n, long long *frac) {
    for (int j = 0; j < n; ++j) {
        crt::Words w;
        crt::each_modulus([&](auto I) { crt::accumulate<decltype(I)::value>(w, y[decltype(I)::value * n + j]); });
        frac[j] = crt::fraction(w);
    }
    return crt::kProduct;
}
