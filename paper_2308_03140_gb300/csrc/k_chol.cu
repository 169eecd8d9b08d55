// FP64 Cholesky factorisation of a batch of matrices on the tensor cores, for the screening solves
// of Eq. (scs) and the log-formula route: the 64-column blocks and the trailing updates are residue
// products (k_crt.cu), only the 64 x 64 diagonal blocks are factored on the FP64 pipe.
//
// A row r of the factor of a positive definite matrix has |L_r|^2 = A_rr, so its scaling exponent is known before
// the factorisation starts and each column block of L becomes residue planes once, for all products
// that read it.  The row of a matrix that is not may be longer, and its products would come back modulo P with any
// pivot: k_solve counts the squares of a row's entries against A_rr and raises ST_SCS_NOT_PD when they
// exceed it by 0.1 % (P leaves 1.8 %; below that the products are exact and the pivot tells).  Panels of kPanel columns; inside a panel, for each block of 64 columns (all launches
// take the whole batch):
//   products   C = A[j:, j] - L[j:, p:j] L[j, p:j]^T          (narrow tiles; not for the first block)
//   k_column   FP64 values of the diagonal block, residues of the rows below
//   k_potrf    its factor and inverse (FP64), the inverse's residues
//   products   L[below, j] = C D^-T
//   k_solve    its FP64 values and its residues in the panel's planes
// then the trailing matrix A22 -= L21 L21^T (lower half) with K = kPanel.  With each 64-column block
// updating the trailing matrix itself, as on the FP64 pipe, that matrix would pass through memory
// once per 64 columns.
#include <algorithm>

#include "crt_dev.cuh"
#include "internal.h"

namespace mbdgb {
namespace {

using crt::kMod;

// exps[b][r] of the rows of the factor, from the diagonal, and left[b][r]: the sum of squares that the row's scaled
// entries may reach, in units of 2^64 (negative for a bad row).
__global__ void k_factor_exponents(const double *A, long long ld, long long mstride, int *exps, float *left) {
    const long long r = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x, b = blockIdx.y;
    if (r >= ld) return;
    const double d = A[b * mstride + r * ld + r];
    const int e = crt::row_exponent(sqrt(d) * (1.0 + 1e-6));   // (the root of a negative diagonal is NaN: a bad row)
    exps[b * ld + r] = e == crt::kBadRow ? e : min(e, 1000);
    const double root = e == crt::kBadRow ? 0.0 : sqrt(d) * crt::pow2(min(e, 1000) - 32);   // below 2^27
    left[b * ld + r] = e == crt::kBadRow ? -1.0f : static_cast<float>(1.001 * root * root);
}

// Two neighbouring entries' residues, bf16 pairs into the planes at `out`.  Returns the sum of their scaled squares in units
// of 2^64, from the upper limbs: to 2^-26 of what a row may reach.
__device__ __forceinline__ float put2(double v0, double v1, double scale, long long plane, __nv_bfloat16 *out) {
    const crt::Limbs l0 = crt::limbs(__double2ll_rn(v0 * scale)), l1 = crt::limbs(__double2ll_rn(v1 * scale));
    crt::each_modulus([&](auto I) {
        constexpr int k = decltype(I)::value;
        const uint32_t f0 = __float_as_uint(crt::residue<k>(l0)), f1 = __float_as_uint(crt::residue<k>(l1));
        *reinterpret_cast<uint32_t *>(out + k * plane) = __byte_perm(f0, f1, 0x7632);
    });
    const float x0 = 65536.0f * l0.l3 + l0.l2, x1 = 65536.0f * l1.l3 + l1.l2;
    return x0 * x0 + x1 * x1;
}
// 2^e (exponents are kept at most 1000: rows below 1e-283 keep fewer bits); zero for bad rows.
__device__ __forceinline__ double row_scale(int e) { return e == crt::kBadRow ? 0.0 : crt::pow2(e); }

__device__ __forceinline__ double warp_sum64(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Two neighbouring entries of a product from its bytes (planes of `plane` bytes).
__device__ __forceinline__ void get2(const uint8_t *y, long long plane, double (&v)[2]) {
    crt::Words s[2];
    crt::each_modulus([&](auto I) {
        constexpr int k = decltype(I)::value;
        const uint32_t p = *reinterpret_cast<const uint16_t *>(y + k * plane);
        crt::accumulate<k>(s[0], p & 255u);
        crt::accumulate<k>(s[1], p >> 8);
    });
    v[0] = static_cast<double>(crt::fraction(s[0])) * crt::kProduct;
    v[1] = static_cast<double>(crt::fraction(s[1])) * crt::kProduct;
}

// Column block j0 (64 columns), a warp per row r = j0 + rr, rr < m: v = A - (product, if Y).  The
// diagonal block's lower half goes back to A; a row below becomes residues (planes [b][kMod][m][64]).
__global__ void __launch_bounds__(256) k_column(double *A, long long ld, long long mstride, int j0, int m,
                                                const uint8_t *Y, const int *fexps, __nv_bfloat16 *planes, int *exps) {
    const int rr = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (rr >= m) return;
    const long long b = blockIdx.y, r = j0 + rr;
    double *a = A + b * mstride + r * ld + j0 + 2 * lane;
    const double2 x = *reinterpret_cast<const double2 *>(a);
    double v[2] = {x.x, x.y};
    if (Y) {
        double p[2];
        const long long plane = 64LL * m;
        get2(Y + b * kMod * plane + 64LL * rr + 2 * lane, plane, p);
        const int er = fexps[b * ld + r];
        const int2 ec = *reinterpret_cast<const int2 *>(fexps + b * ld + j0 + 2 * lane);
        v[0] -= crt::scaled_down(p[0], er, ec.x);
        v[1] -= crt::scaled_down(p[1], er, ec.y);
    }
    if (rr < 64) {
        if (Y) {
            if (2 * lane <= rr) a[0] = v[0];
            if (2 * lane + 1 <= rr) a[1] = v[1];
        }
        return;
    }
    const double ss = warp_sum64(v[0] * v[0] + v[1] * v[1]);
    int e;
    if (ss > 1e-280 && ss < 1e280) {
        e = crt::row_exponent(sqrt(ss));
    } else {   // an upper bound of the norm serves: 8 times the largest entry
        double mx = fmax(fabs(v[0]), fabs(v[1]));   // (drops a NaN beside a number)
        if (!(mx <= crt::kMaxDouble / 16) || isnan(v[0]) || isnan(v[1])) mx = CUDART_INF;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        e = crt::row_exponent(8.0 * mx);
    }
    e = e == crt::kBadRow ? e : min(e, 1000);
    if (e == crt::kBadRow) v[0] = v[1] = 0.0;
    if (lane == 0) exps[b * m + rr] = e;
    const long long plane = 64LL * m;
    put2(v[0], v[1], row_scale(e), plane, planes + b * kMod * plane + 64LL * rr + 2 * lane);
}

// Row r = j0 + 64 + rr of the solved block, a warp per row: FP64 values from the product's bytes, and
// residues at the row's exponent in the panel's planes ([b][kMod][ld][pitch], columns from kcol).  The squares of the scaled
// entries are taken from left[b][r], which this launch alone touches: in FP32, whose 1e-7 a block of columns is far
// inside the 0.1 %, as FP64 sums over the warp would take the pipe that bounds this kernel.
__global__ void __launch_bounds__(256) k_solve(double *A, long long ld, long long mstride, int j0, int m,
                                               const uint8_t *Y, const int *rexps, long long rstride, const int *dexps,
                                               const int *fexps, __nv_bfloat16 *planes, int pitch, int kcol, float *left,
                                               int *status) {
    const int rr = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (rr >= m) return;
    const long long b = blockIdx.y, r = j0 + 64 + rr, plane = 64LL * m;
    double v[2];
    get2(Y + b * kMod * plane + 64LL * rr + 2 * lane, plane, v);
    const int er = rexps[b * rstride + rr];
    const int2 ec = *reinterpret_cast<const int2 *>(dexps + b * 64 + 2 * lane);
    v[0] = crt::scaled_down(v[0], er, ec.x);
    v[1] = crt::scaled_down(v[1], er, ec.y);
    *reinterpret_cast<double2 *>(A + b * mstride + r * ld + j0 + 2 * lane) = make_double2(v[0], v[1]);
    const int e = fexps[b * ld + r];
    const bool fine = fabs(v[0]) <= crt::kMaxDouble && fabs(v[1]) <= crt::kMaxDouble;
    if (e == crt::kBadRow || !fine) v[0] = v[1] = 0.0;   // (a factorisation that has failed)
    const long long pp = ld * pitch;
    float used = put2(v[0], v[1], row_scale(e), pp, planes + b * kMod * pp + r * pitch + kcol + 2 * lane);
    if (!fine) used = CUDART_INF_F;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) used += __shfl_xor_sync(0xffffffffu, used, o);
    if (lane == 0) {
        const float rest = left[b * ld + r] - used;
        left[b * ld + r] = rest;
        if (!(rest >= 0.0f)) atomicOr(status, ST_SCS_NOT_PD);
    }
}

// 1 / d, d a normal number: two Newton steps from the hardware's approximation (2^-20 or better), after which only the last
// rounding is left, so that all but a few quotients are the division's.  (Diagonals beyond 1e+-280, the inverses of
// polarizabilities in bohr^3, are not served, here and in the exponents.)
__device__ __forceinline__ double reciprocal(double d) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;\n" : "=d"(y) : "d"(d));
    y = fma(y, fma(-d, y, 1.0), y);
    return fma(y, fma(-d, y, 1.0), y);
}

// Factor and inverse of a 64 x 64 diagonal block.  A cluster of four CTAs takes one matrix: each
// factors the block by itself (its 45e3 multiply-adds take 11 us of an SM's FP64 pipe, exchanging columns
// would take longer) and inverts every fourth column, so that the inverse, as much work again,
// takes a quarter of that.  The factorisation keeps the block in registers (thread (ty, tx): rows
// ty + 16 a, columns tx + 16 c) in the form L D L^T, one reciprocal and one barrier a column: the
// warp that holds the next column updates it first, forms its pivot's reciprocal and stores the
// column before the rest of its update.  Then L_ij = a_ij / sqrt(d_j).  The inverse's rows are
// turned into residues for the product that solves the rows below (planes [b][kMod][64][64]).
__global__ void __cluster_dims__(4, 1, 1) __launch_bounds__(256)
    k_potrf(double *A, long long ld, long long mstride, double *dinv, long long dstride, int *status,
            __nv_bfloat16 *planes, int *exps) {
    __shared__ double S[64][65];        // the factor; then the inverse's columns of this CTA
    __shared__ double col[2][64], row[2][64];   // column j, and divided by its pivot
    __shared__ double piv[64], inv[64], part[64];
    __shared__ int bad;
    const int q = blockIdx.x & 3;       // rank in the cluster
    const long long b = blockIdx.x >> 2;
    double *Ab = A + b * mstride;
    const int t = threadIdx.x, ty = t & 15, tx = t >> 4;   // a warp holds two columns' rows
    if (t == 0) bad = 0;
    double a[4][4];   // a[i][c]: row ty + 16 i, column tx + 16 c; lower half
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c <= i; ++c) a[i][c] = (tx + 16 * c <= ty + 16 * i) ? Ab[(ty + 16 * i) * ld + tx + 16 * c] : 0.0;
    // every CTA of the cluster has read the block before one writes its factor
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    // The pivot of column j = 16 cb + jx and its reciprocal, in the warp that holds the column; then the
    // column itself to shared memory, by its owners (half the warp).
    auto pivot = [&](auto CB, int jx, double &r) {
        constexpr int cb = decltype(CB)::value;
        double d = __shfl_sync(0xffffffffu, a[cb][cb], (t & 16) | jx);
        const bool ok = d > 0.0;
        d = ok ? d : 1.0;
        r = reciprocal(d);
        if (tx == jx && ty == jx) {
            if (!ok) bad = 1;
            piv[16 * cb + jx] = d;
        }
    };
    auto publish = [&](auto CB, int jx, double r) {
        constexpr int cb = decltype(CB)::value;
        const int p = jx & 1;   // the parity of j
        if (tx != jx) return;
#pragma unroll
        for (int i = cb; i < 4; ++i) {
            if (i > cb || ty > jx) {
                col[p][ty + 16 * i] = a[i][cb];
                row[p][ty + 16 * i] = a[i][cb] * r;
            }
        }
    };
    auto blocks = [&](auto CB) {   // columns 16 cb .. 16 cb + 15
        constexpr int cb = decltype(CB)::value;
        for (int jx = 0; jx < 16; ++jx) {
            const int j = 16 * cb + jx, p = j & 1;
            __syncthreads();   // column j is there; the buffer of column j + 1 is free
            double x[4], w[4];
#pragma unroll
            for (int i = cb; i < 4; ++i) {
                x[i] = ty + 16 * i > j ? col[p][ty + 16 * i] : 0.0;
                w[i] = tx + 16 * i > j ? row[p][tx + 16 * i] : 0.0;
            }
            // the next pivot first, then its column: every FP64 instruction of the warp that holds them is
            // 64 cycles of the chain
            a[cb][cb] -= x[cb] * w[cb];
            const bool owner = jx < 15 && tx >> 1 == (jx + 1) >> 1;
            double r = 0.0;
            if (owner) pivot(CB, jx + 1, r);
#pragma unroll
            for (int i = cb + 1; i < 4; ++i) a[i][cb] -= x[i] * w[cb];
            if (owner) publish(CB, jx + 1, r);
#pragma unroll
            for (int c = cb + 1; c < 4; ++c)
#pragma unroll
                for (int i = c; i < 4; ++i) a[i][c] -= x[i] * w[c];
            if constexpr (cb < 3) {
                if (jx == 15 && tx < 2) {
                    pivot(std::integral_constant<int, cb + 1>{}, 0, r);
                    publish(std::integral_constant<int, cb + 1>{}, 0, r);
                }
            }
        }
    };
    if (tx < 2) {
        double r;
        pivot(std::integral_constant<int, 0>{}, 0, r);
        publish(std::integral_constant<int, 0>{}, 0, r);
    }
    blocks(std::integral_constant<int, 0>{});
    blocks(std::integral_constant<int, 1>{});
    blocks(std::integral_constant<int, 2>{});
    blocks(std::integral_constant<int, 3>{});
    __syncthreads();
    if (t < 64) {
        const double s = sqrt(piv[t]);
        S[t][t] = s;
        inv[t] = 1.0 / s;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c <= i; ++c) {
            const int r = ty + 16 * i, k = tx + 16 * c;
            if (k < r) S[r][k] = a[i][c] * inv[k];
        }
    __syncthreads();
    for (int e = t; e < 1024; e += 256) {   // every fourth row of the factor back to A
        const int r = 4 * (e >> 6) + q, c = e & 63;
        if (c <= r) Ab[r * ld + c] = S[r][c];
    }
    // Inverse by columns: half a warp per column k = 4 g + q, lane ty its rows ty + 16 i.
    const int k = 4 * tx + q;
    double y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) y[i] = ty + 16 * i == k ? 1.0 : 0.0;
#pragma unroll
    for (int ib = 0; ib < 4; ++ib) {
        for (int jx = 0; jx < 16; ++jx) {
            const int j = 16 * ib + jx;
            if (j < 4 * (tx & ~1)) continue;   // above both of the warp's columns (uniform in the warp)
            const double v = __shfl_sync(0xffffffffu, y[ib] * inv[j], (threadIdx.x & 16) | jx);
            if (ty == jx) y[ib] = v;
#pragma unroll
            for (int i = ib; i < 4; ++i) {
                const int r = ty + 16 * i;
                if (r > j) y[i] -= S[r][j] * v;
            }
        }
    }
    // its rows' norms over the cluster, their exponents and residues
    __shared__ double sq[64][17];
#pragma unroll
    for (int i = 0; i < 4; ++i) sq[ty + 16 * i][tx] = y[i] * y[i];
    double *Db = dinv + b * dstride;
#pragma unroll
    for (int i = 0; i < 4; ++i) Db[(ty + 16 * i) * 64 + k] = ty + 16 * i >= k ? y[i] : 0.0;
    __syncthreads();
    if (t < 64) {
        double s = 0.0;
        for (int c = 0; c < 16; ++c) s += sq[t][c];
        part[t] = s;
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    __shared__ int re[64];
    if (t < 64) {
        double s = 0.0;
        const uint32_t mine = static_cast<uint32_t>(__cvta_generic_to_shared(&part[t]));
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            uint32_t addr;
            double v;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(addr) : "r"(mine), "r"(c));
            asm volatile("ld.shared::cluster.f64 %0, [%1];\n" : "=d"(v) : "r"(addr));
            s += v;
        }
        // the squares over- or underflow only for factors beyond 1e140: those rows are marked bad
        const int e = s > 1e-280 && s < 1e280 ? min(crt::row_exponent(sqrt(s)), 1000) : crt::kBadRow;
        re[t] = e;
        if (q == 0) exps[b * 64 + t] = e;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = ty + 16 * i, e = re[r];
        const crt::Limbs l = crt::limbs(__double2ll_rn((r >= k && e != crt::kBadRow ? y[i] : 0.0) * row_scale(e)));
        __nv_bfloat16 *o = planes + b * kMod * 4096 + r * 64 + k;
        crt::each_modulus([&](auto I) {
            constexpr int mi = decltype(I)::value;
            o[mi * 4096] = __ushort_as_bfloat16(static_cast<unsigned short>(__float_as_uint(crt::residue<mi>(l)) >> 16));
        });
    }
    if (t == 0 && q == 0 && bad) atomicOr(status, ST_SCS_NOT_PD);
    // no CTA leaves while another may still read its part[]
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// Columns of a panel.  Its planes take 480 ld kPanel bytes for 16 matrices; each panel passes the
// trailing matrix through memory once.
constexpr int kPanel = 512;

inline size_t al(size_t b) { return (b + 255) / 256 * 256; }

struct Layout {
    long long panel, rows, inverse, exps, rexps, dexps, left, bytes, total;   // offsets
};
Layout layout(long long ld, int batch, const ScratchLimits &lim) {
    Layout l;
    size_t p = 0;
    auto take = [&](size_t n) {
        const size_t at = p;
        p += al(n);
        return static_cast<long long>(at);
    };
    const size_t z = static_cast<size_t>(kMod) * batch;
    l.panel = take(2 * z * ld * std::min<long long>(kPanel, ld));
    l.rows = take(2 * z * ld * 64);
    l.inverse = take(2 * z * 4096);
    l.exps = take(4 * static_cast<size_t>(batch) * ld);
    l.rexps = take(4 * static_cast<size_t>(batch) * ld);
    l.dexps = take(4 * static_cast<size_t>(batch) * 64);
    l.left = take(4 * static_cast<size_t>(batch) * ld);
    const size_t m = ld > kPanel ? static_cast<size_t>(ld) - kPanel : 0, whole = kMod * m * m;
    const size_t strip = kMod * m * std::min<size_t>(m, lim.strip);
    l.bytes = take(std::max<size_t>(z * ld * 64, std::min<size_t>(whole * batch, std::max<size_t>(lim.trailing, strip))));
    l.total = static_cast<long long>(p);
    return l;
}

}  // namespace

size_t cholesky_crt_bytes(long long ld, int batch, const ScratchLimits &lim) {
    return static_cast<size_t>(layout(ld, batch, lim).total);
}

cudaError_t cholesky_crt(double *A, long long ld, long long mstride, int batch, double *dinv, void *work, int *status,
                         cudaStream_t s, const ScratchLimits &lim) {
    const Layout l = layout(ld, batch, lim);
    char *w = static_cast<char *>(work);
    auto *panel = reinterpret_cast<__nv_bfloat16 *>(w + l.panel), *rows = reinterpret_cast<__nv_bfloat16 *>(w + l.rows),
         *inverse = reinterpret_cast<__nv_bfloat16 *>(w + l.inverse);
    int *exps = reinterpret_cast<int *>(w + l.exps), *rexps = reinterpret_cast<int *>(w + l.rexps),
        *dexps = reinterpret_cast<int *>(w + l.dexps);
    float *left = reinterpret_cast<float *>(w + l.left);
    uint8_t *Y = reinterpret_cast<uint8_t *>(w + l.bytes);
    const size_t ybytes = static_cast<size_t>(l.total - l.bytes);
    const int nb = static_cast<int>(ld / kTile), pitch = static_cast<int>(std::min<long long>(kPanel, ld));
    const long long plane = ld * pitch;
    // rows r0 .. r0 + n - 1 of `count` matrices' planes from matrix b0, K columns, as an operand
    auto panel_rows = [&](int b0, int count, long long r0, long long n, int K) {
        CrtOperand o{};
        o.shape.rows = o.shape.out_rows = static_cast<int>(n);
        o.shape.K = K;
        o.shape.batch = count;
        o.shape.pitch = pitch;
        o.plane = plane;
        o.exp_stride = ld;
        o.planes = panel + b0 * kMod * plane + r0 * pitch;
        o.exps = exps + b0 * ld + r0;
        return o;
    };
    auto block = [&](__nv_bfloat16 *planes, int *e, int n) {   // n x 64 planes of every matrix
        CrtOperand o{};
        o.shape.rows = o.shape.out_rows = n;
        o.shape.K = 64;
        o.shape.batch = batch;
        o.shape.pitch = 64;
        o.plane = 64LL * n;
        o.exp_stride = n;
        o.planes = planes;
        o.exps = e;
        return o;
    };
    count_launches(1);
    k_factor_exponents<<<dim3(static_cast<unsigned>((ld + 255) / 256), batch), 256, 0, s>>>(A, ld, mstride, exps, left);
    cudaError_t e = cudaSuccess;
    for (long long p0 = 0; p0 < ld; p0 += kPanel) {
        const long long p1 = std::min<long long>(ld, p0 + kPanel);
        for (long long j0 = p0; j0 < p1; j0 += 64) {
            const int m = static_cast<int>(ld - j0), kc = static_cast<int>(j0 - p0);
            if (kc) {
                e = crt_products(panel_rows(0, batch, j0, m, kc), panel_rows(0, batch, j0, 64, kc), m, 0, Y, status, s);
                if (e != cudaSuccess) return e;
            }
            count_launches(2);
            k_column<<<dim3((m + 7) / 8, batch), 256, 0, s>>>(A, ld, mstride, static_cast<int>(j0), m, kc ? Y : nullptr,
                                                              exps, rows, rexps);
            k_potrf<<<4 * batch, 256, 0, s>>>(A + j0 * ld + j0, ld, mstride, dinv + (j0 / kTile) * 4096LL,
                                              static_cast<long long>(nb) * 4096, status, inverse, dexps);
            const int below = m - 64;
            if (below <= 0) continue;
            CrtOperand c = block(rows, rexps, m);   // the rows below the diagonal block
            c.shape.rows = c.shape.out_rows = below;
            c.planes += 64 * 64;
            c.exps += 64;
            e = crt_products(c, block(inverse, dexps, 64), below, 0, Y, status, s);
            if (e != cudaSuccess) return e;
            count_launches(1);
            k_solve<<<dim3((below + 7) / 8, batch), 256, 0, s>>>(A, ld, mstride, static_cast<int>(j0), below, Y, rexps + 64,
                                                                m, dexps, exps, panel, pitch, kc, left, status);
        }
        const long long m = ld - p1;
        if (m <= 0) continue;
        const int K = static_cast<int>(p1 - p0);
        const size_t one = kMod * static_cast<size_t>(m) * m;
        const int group = static_cast<int>(std::min<size_t>(batch, ybytes / one));
        for (int b0 = 0; b0 < batch; b0 += std::max(group, 1)) {
            const int g = std::min(std::max(group, 1), batch - b0);
            // columns of the lower half in strips when one matrix's bytes are too many
            const long long width = group ? m : std::max<long long>(256, static_cast<long long>(ybytes / (kMod * m)) / 256 * 256);
            for (long long c0 = 0; c0 < m; c0 += width) {
                const long long n = std::min(width, m - c0), r0 = p1 + c0;
                double *C = A + b0 * mstride + r0 * ld + r0;
                const CrtResult r{-1.0, 1.0, C, C, nullptr, ld, ld, 0, mstride, mstride, 0, 0, 0, 2};
                e = crt_multiply(panel_rows(b0, g, r0, m - c0, K), panel_rows(b0, g, r0, n, K), r, Y, status, s);
                if (e != cudaSuccess) return e;
            }
        }
    }
    return cudaGetLastError();
}

}  // namespace mbdgb
