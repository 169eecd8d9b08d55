// Arithmetic of the FP64 products on the bf16 tensor cores by residues (k_crt.cu), host and
// device: integers of up to 58 bits, their residues modulo 15 small coprime moduli, and the way
// back (Chinese remainder theorem; the scheme of Ozaki, Uchino and Imamura, arXiv 2504.08009, with
// bf16 operands and FP32 accumulation in place of INT8).
//
// A row a of the left operand is scaled by a power of two and rounded to integers x = rint(a 2^e)
// with |x|_2 < sqrt(P/2), P the product of the moduli; likewise a column b of the right one.
// Then |x.y| < P/2, so x.y is known from its residues: for each modulus m the tensor cores
// sum products of residues in [-128, 128] (exact in bf16: 8 bits), 1024 of them at a time, so that
// every partial sum is an integer of at most 2^24 and exact in FP32.  What is lost is only the rounding of x
// and y: an error of about 0.4 2^-kRowBits |a| |b| in a.b, against about 0.2 2^-52 |a| |b| for an
// FP64 sum of random terms, whose roundings grow with their number.  That is relative to the rows' norms: where one
// entry dominates a row and meets a small one, so that |a.b| is far below |a| |b|, an FP64 sum keeps more
// bits of a.b (entries 1e-8 of their rows: 2e-16 against 2e-11).  The matrices here are summed into traces and
// contracted with rows of their own size, and over the sizes the library is timed on the results' errors against
// 64-bit eigenvalues are what they were on the FP64 pipe.
#pragma once
#include <cmath>
#include <cstdint>
#include <type_traits>

#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace mbdgb {
namespace crt {

constexpr int kMod = 15;   // P = 2^117.78; with 14 moduli (2^110.2) the small entries of a row with one
                           // large entry would keep fewer bits than an FP64 sum gives them
constexpr int kModuli[kMod] = {256, 255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197};
constexpr int kRowBits = 58;   // scaled rows have |x|_2 <= 0.65 * 2^(kRowBits + 1) < sqrt(P/2) = 2^58.39
constexpr int kStageK = 64;    // K per shared-memory stage (128 bytes of bf16)
constexpr int kChunk = 16;     // stages per FP32 accumulation: 1024 products of at most 2^14

constexpr int mod_pow2(int k, int m) {   // 2^k mod m in [-m/2, m/2]
    int r = 1 % m;
    for (int i = 0; i < k; ++i) r = (2 * r) % m;
    return 2 * r > m ? r - m : r;
}
constexpr int inverse_of_rest(int i) {   // (P / m_i)^-1 mod m_i in [0, m_i)
    const int m = kModuli[i];
    int rest = 1;
    for (int j = 0; j < kMod; ++j)
        if (j != i) rest = rest * (kModuli[j] % m) % m;
    for (int q = 1; q < m; ++q)
        if (rest * q % m == 1) return q;
    return 0;
}
constexpr uint32_t weight_word(int i, int w) {   // word w (0 lowest) of round(2^96 / m_i)
    const uint64_t m = static_cast<uint64_t>(kModuli[i]);
    uint64_t d[3] = {0, 0, 0}, rem = 1;
    for (int k = 2; k >= 0; --k) {
        rem <<= 32;
        d[k] = rem / m;
        rem %= m;
    }
    if (2 * rem >= m) {   // no carry out: 2^96 / m has fewer than 96 bits
        for (int k = 0; k < 3; ++k) {
            d[k] = (d[k] + 1) & 0xffffffffull;
            if (d[k]) break;
        }
    }
    return static_cast<uint32_t>(d[w]);
}
constexpr double product_scaled() {   // P 2^-64, rounded once
    unsigned __int128 p = 1;
    for (int i = 0; i < kMod; ++i) p *= static_cast<unsigned>(kModuli[i]);
    return static_cast<double>(p) / 18446744073709551616.0;
}

// The constants of modulus I as scalars, so that unrolled device code holds them as immediates.
template <int I>
struct Modulus {
    static constexpr float m = static_cast<float>(kModuli[I]), inv = 1.0f / static_cast<float>(kModuli[I]);
    static constexpr float c1 = static_cast<float>(mod_pow2(16, kModuli[I])),
                           c2 = static_cast<float>(mod_pow2(32, kModuli[I])),
                           c3 = static_cast<float>(mod_pow2(48, kModuli[I]));
    static constexpr float back = static_cast<float>(inverse_of_rest(I));
    static constexpr uint32_t w0 = weight_word(I, 0), w1 = weight_word(I, 1), w2 = weight_word(I, 2);
};
constexpr double kProduct = product_scaled();

// f(integral_constant<int, I>) for I = 0 .. kMod - 1.
template <int I = 0, class F>
__host__ __device__ __forceinline__ void each_modulus(F &&f) {
    if constexpr (I < kMod) {
        f(std::integral_constant<int, I>{});
        each_modulus<I + 1>(f);
    }
}

__host__ __device__ __forceinline__ float fma32(float a, float b, float c) {
#ifdef __CUDA_ARCH__
    return __fmaf_rn(a, b, c);
#else
    return std::fmaf(a, b, c);
#endif
}
__host__ __device__ __forceinline__ float add32(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fadd_rn(a, b);
#else
    volatile float s = a + b;
    return s;
#endif
}

constexpr float kMagic = 12582912.0f;   // 1.5 * 2^23: adding and taking it away rounds to an integer
// r mod m in [-m/2 - 1, m/2 + 1] for an integer |r| <= 2^24: r/m is known to 1/m, so the rounded
// quotient is off by at most that.
__host__ __device__ __forceinline__ float reduce(float r, float m, float inv) {
    const float q = add32(fma32(r, inv, kMagic), -kMagic);
    return fma32(-m, q, r);
}

// The exponent e of a row of 2-norm `norm`: 2^e norm <= 0.65 * 2^(kRowBits + 1).  0 for a zero row;
// kBadRow for one that is not finite, whose products are NaN.
constexpr int kBadRow = 0x7fffffff;
constexpr double kMaxDouble = 1.7976931348623157e308;
__host__ __device__ __forceinline__ int row_exponent(double norm) {
    if (!(norm <= kMaxDouble)) return kBadRow;
    if (norm == 0.0) return 0;
    int x;
    const double f = frexp(norm, &x);   // norm = f 2^x, f in [0.5, 1)
    return kRowBits - x + (f <= 0.65 ? 1 : 0);   // -966 .. 1132
}
__host__ __device__ __forceinline__ double pow2(int e) {   // 2^e, |e| <= 1022
#ifdef __CUDA_ARCH__
    return __longlong_as_double(static_cast<long long>(e + 1023) << 52);
#else
    return std::ldexp(1.0, e);
#endif
}

// Balanced 16-bit limbs of x, |x| <= 2^60: x = l0 + l1 2^16 + l2 2^32 + l3 2^48.
struct Limbs {
    float l0, l1, l2, l3;
};
__host__ __device__ __forceinline__ Limbs limbs(long long x) {
    const int a = static_cast<short>(x);
    x = (x - a) >> 16;
    const int b = static_cast<short>(x);
    x = (x - b) >> 16;
    const int c = static_cast<short>(x);
    x = (x - c) >> 16;
    return {static_cast<float>(a), static_cast<float>(b), static_cast<float>(c), static_cast<float>(static_cast<int>(x))};
}
// x mod m_I: the limbs' sum is below 2^15 + 2 * 2^22 + 2^19 < 2^24 and exact.
template <int I>
__host__ __device__ __forceinline__ float residue(const Limbs &l) {
    using M = Modulus<I>;
    return reduce(fma32(l.l3, M::c3, fma32(l.l2, M::c2, fma32(l.l1, M::c1, l.l0))), M::m, M::inv);
}

// What the product's residue r (|r| <= m/2 + 1) is stored as: r (P/m)^-1 mod m in [0, m).
__host__ __device__ __forceinline__ float stored(float r, float m, float inv, float back) {
    const float y = reduce(r * back, m, inv);   // |r back| < 2^16
    return y < 0.0f ? y + m : y;
}

// From the stored residues to the integer: sum_i y_i / m_i is x.y / P up to an integer.  It is summed
// in units of 2^-96 in three words (the products below 2^40, their sums below 2^44), of which the
// upper 64 bits as a signed fraction times P are the result, rounded to P 2^-64, which is less than
// the rounding of the rows left.
struct Words {
    unsigned long long s0 = 1ull << 31, s1 = 0, s2 = 0;   // (the first rounds: a cut would bias every entry alike)
};
template <int I>
__host__ __device__ __forceinline__ void accumulate(Words &w, uint32_t y) {
    using M = Modulus<I>;
    w.s0 += static_cast<unsigned long long>(y) * M::w0;
    w.s1 += static_cast<unsigned long long>(y) * M::w1;
    w.s2 += static_cast<unsigned long long>(y) * M::w2;
}
__host__ __device__ __forceinline__ long long fraction(const Words &w) {
    return static_cast<long long>((w.s2 << 32) + w.s1 + (w.s0 >> 32));
}

}  // namespace crt
}  // namespace mbdgb
