// Gradient of a cell's energy (periodic_mbd_grad of k_periodic.cu, which has the formulas) with its sums over
// atoms and Bloch vectors as products on the tensor cores.
//
// With z_ij the symmetric part of w Z_q's block (w = kw zscale / (4 nkt)) and c_i = omega_bar_i sqrt(abar0_i):
// Reciprocal space: everything follows from U_e,j(G) = sum_i c_i conj(z_e,ij) conj(S_iG) for the six components e,
// one complex product of 6N x N by N x nG for each Bloch vector; an atom j and a vector G are then left with 100
// operations where every pair and G had them.
// Real space: at image r = r0 + o A of a pair (r0 the first one) the derivatives of the tensors meet
//   A_e(o) = sum_q Re y_e e^{-i q.oA},  B_de(o) = sum_q q_d Im y_e e^{-i q.oA},  y = conj(z) e^{-i q.r0},
// real products of the pairs' rows y (2 nk entries) with one table of the image offsets, so that the radial functions
// are evaluated once for all Bloch vectors.
// Both are formed FP64-accurately by residues (k_crt.cu); the mixed modes' reciprocal sums stay with the FP32 kernel.
// On the FP64 pipe, a thread per pair and Bloch vector, the pass took 20.1 ms for the 96-atom cell
// (automatic Ewald split, 64 Bloch vectors), 2.0 so; the 256-atom cell's real space took 28 ms, 3.7 so.
#include <algorithm>

#include "cell_pairs.cuh"
#include "internal.h"
#include "pair_math.cuh"

namespace mbdgb {
namespace {

using namespace pairs;
using namespace cellpairs;

__device__ __forceinline__ double coupling(const AtomBufs &b, int i) { return b.ombar[i] * sqrt(b.abar0[i]); }
// Rows and columns of component e (xx, yy, zz, xy, xz, yz).
__device__ __forceinline__ int comp_row(int e) { return e < 3 ? e : (e == 5 ? 1 : 0); }
__device__ __forceinline__ int comp_col(int e) { return e < 3 ? e : (e == 3 ? 1 : 2); }

// Left rows (e, j) of Bloch vector k0 + blockIdx.z: entries i, w c_i conj(z_e,ij) with z_ij of the block (min, max) (planar;
// zero imaginary parts for i = j, whose block is Hermitian); [z][2][6 N][ldn].
__global__ void k_grad_left(AtomBufs b, PeriodicBufs p, const double *Z, long long ld, double zscale, int k0, int ldn,
                            double *left) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y % b.N, e = blockIdx.y / b.N, z = blockIdx.z, kq = k0 + z;
    if (i >= ldn) return;
    double re = 0.0, im = 0.0;
    if (i < b.N) {
        const double *Zr = Z + static_cast<long long>(kq) * 2 * ld * ld, *Zi = Zr + ld * ld;
        const long long lo = 3LL * min(i, j), hi = 3LL * max(i, j), ra = comp_row(e), rb = comp_col(e);
        const long long o1 = (lo + ra) * ld + hi + rb, o2 = (lo + rb) * ld + hi + ra;
        const double w = 0.125 * zscale / p.nkt * p.kw[kq] * coupling(b, i);
        re = w * (Zr[o1] + Zr[o2]);
        im = w * (Zi[o1] + Zi[o2]);
        im = i < j ? -im : (i > j ? im : 0.0);
    }
    double *l = left + ((z * 12LL + e) * b.N + j) * ldn + i;
    l[0] = re;
    l[6LL * b.N * ldn] = im;
}

// Right rows G: entries i, conj(S_iG) (planar; zero beyond the Bloch vector's list); [z][2][rows][ldn].
__global__ void k_grad_right(PeriodicBufs p, int N, int k0, int rows, int ldn, double *right) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, g = blockIdx.y, z = blockIdx.z, kq = k0 + z;
    if (i >= ldn) return;
    double2 s = make_double2(0.0, 0.0);
    if (i < N && g < p.gcount[kq]) s = p.S[static_cast<long long>(p.glist[static_cast<long long>(kq) * p.maxG + g]) * N + i];
    double *r = right + (z * 2LL * rows + g) * ldn + i;
    r[0] = s.x;
    r[static_cast<long long>(rows) * ldn] = -s.y;
}

// What U gives atom j = 4 blockIdx.x + warp at Bloch vector k0 + blockIdx.y.
__global__ void __launch_bounds__(128) k_grad_recip(AtomBufs b, PeriodicBufs p, int k0, const double *U, int ldg, double *g_c,
                                                    double *gR, double *gA) {
    const int lane = threadIdx.x & 31, j = blockIdx.x * 4 + (threadIdx.x >> 5), z = blockIdx.y, kq = k0 + z;
    if (j >= b.N) return;
    const CellGeom &c = p.cell;
    const int cnt = p.gcount[kq];
    const int *gl = p.glist + static_cast<long long>(kq) * p.maxG;
    const double q[3] = {p.kq[3 * kq], p.kq[3 * kq + 1], p.kq[3 * kq + 2]};
    const double *Uj = U + (z * 12LL * b.N + j) * ldg;
    const long long comp = static_cast<long long>(b.N) * ldg, im = 6 * comp;
    const double pre = 4.0 * kPi / c.vol, damp = 0.25 / (c.gamma * c.gamma);
    double sum[13];   // su, M1, M2
#pragma unroll
    for (int t = 0; t < 13; ++t) sum[t] = 0.0;
    for (int g = lane; g < cnt; g += 32) {
        const int gi = gl[g];
        const double *G = p.G + 3LL * gi;
        const double2 s2 = p.S[static_cast<long long>(gi) * b.N + j];
        const double k[3] = {G[0] + q[0], G[1] + q[1], G[2] + q[2]};
        const double Gr[3] = {G[0], G[1], G[2]};
        const double sx = s2.x, sy = s2.y;
        const double k2 = k[0] * k[0] + k[1] * k[1] + k[2] * k[2], ik2 = 1.0 / k2;
        const double cf = pre * exp(-k2 * damp) * ik2;
        double us[6], vs[6];
#pragma unroll
        for (int e = 0; e < 6; ++e) {
            const double ur = Uj[e * comp + g], ui = Uj[im + e * comp + g];
            us[e] = ur * sx - ui * sy;
            vs[e] = ur * sy + ui * sx;
        }
        const double uk[3] = {us[0] * k[0] + us[3] * k[1] + us[4] * k[2], us[3] * k[0] + us[1] * k[1] + us[5] * k[2],
                         us[4] * k[0] + us[5] * k[1] + us[2] * k[2]};
        const double kuk = k[0] * uk[0] + k[1] * uk[1] + k[2] * uk[2];
        const double kvk = k[0] * (vs[0] * k[0] + 2.0 * (vs[3] * k[1] + vs[4] * k[2])) + k[1] * (vs[1] * k[1] + 2.0 * vs[5] * k[2]) +
                      vs[2] * k[2] * k[2];
        const double cv = cf * kvk, f2 = kuk * (2.0 * ik2 + 2.0 * damp);
        sum[0] += cf * kuk;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            sum[1 + d] += Gr[d] * cv;
            const double De = cf * (2.0 * uk[d] - f2 * k[d]);
#pragma unroll
            for (int dd = 0; dd < 3; ++dd) sum[4 + 3 * dd + d] += k[dd] * De;
        }
    }
#pragma unroll
    for (int t = 0; t < 13; ++t) sum[t] = warp_sum(sum[t]);
    if (lane) return;
    const double cj = coupling(b, j);
    atomicAdd(&g_c[j], 2.0 * sum[0]);
    for (int d = 0; d < 3; ++d) atomicAdd(&gR[3 * j + d], -2.0 * cj * sum[1 + d]);
    for (int k = 0; k < 3; ++k) {
        const double f = b.R[3 * j] * c.Ainv[k] + b.R[3 * j + 1] * c.Ainv[3 + k] + b.R[3 * j + 2] * c.Ainv[6 + k];
        for (int d = 0; d < 3; ++d) {
            double t = -c.Ainv[3 * d + k] * sum[0] + 2.0 * f * sum[1 + d];
            for (int e = 0; e < 3; ++e) t -= sum[4 + 3 * d + e] * c.Ainv[3 * e + k];
            atomicAdd(&gA[3 * k + d], cj * t);
        }
    }
}

// Pair `at` (its place in the list of pairs) and whether it is one.
__device__ __forceinline__ Pair pair_at(const AtomBufs &b, int ntile, long long at) {
    int I, J;
    tile_pair(static_cast<int>(at / 256), ntile, I, J);
    const int t = static_cast<int>(at % 256), ty = t / kQT, tx = t % kQT;
    Pair p;
    p.i = I * kQT + ty;
    p.j = J * kQT + tx;
    p.valid = p.i < b.N && p.j < b.N && (I < J || ty <= tx);
    for (int e = 0; e < 3; ++e) p.x[e] = p.valid ? b.R[3 * p.j + e] - b.R[3 * p.i + e] : 0.0;
    return p;
}

// Rows (pair, e) of y: entries q, real parts and then imaginary ones; [pairs][6][2 nk].  A thread per pair and q, q fastest.
__global__ void __launch_bounds__(256) k_grad_rows(AtomBufs b, PeriodicBufs p, const double *Z, long long ld, double zscale,
                                                   int ntile, long long pair0, long long pairs, double *rows) {
    const long long id = blockIdx.x * 256LL + threadIdx.x;
    const int kq = static_cast<int>(id % p.nk);
    const long long at = id / p.nk;
    if (at >= pairs) return;
    const Pair pr = pair_at(b, ntile, pair0 + at);
    double *y = rows + at * 12 * p.nk + kq;
    if (!pr.valid) {
        for (int e = 0; e < 12; ++e) y[static_cast<long long>(e) * p.nk] = 0.0;
        return;
    }
    const CellGeom &c = p.cell;
    int lo[3], hi[3];
    image_box(c, pr.x, lo, hi);
    double t = 0.0;
    for (int e = 0; e < 3; ++e)
        t += p.kq[3 * kq + e] * (pr.x[e] + lo[0] * c.A[e] + lo[1] * c.A[3 + e] + lo[2] * c.A[6 + e]);
    double sn, cs;
    sincos(-t, &sn, &cs);
    const double w = 0.125 * zscale / p.nkt * p.kw[kq] * (pr.i == pr.j ? 1.0 : 2.0);
    const double *Zr = Z + static_cast<long long>(kq) * 2 * ld * ld, *Zi = Zr + ld * ld;
#pragma unroll
    for (int e = 0; e < 6; ++e) {
        const long long ra = comp_row(e), rb = comp_col(e);
        const long long o1 = (3LL * pr.i + ra) * ld + 3LL * pr.j + rb, o2 = (3LL * pr.i + rb) * ld + 3LL * pr.j + ra;
        const double zr = w * (Zr[o1] + Zr[o2]), zi = w * (Zi[o1] + Zi[o2]);
        y[2LL * e * p.nk] = zr * cs + zi * sn;
        y[(2LL * e + 1) * p.nk] = zr * sn - zi * cs;
    }
}

// The table's columns as rows: A_e(o) and B_xe .. B_ze(o) take (Re, -Im) and q_d (Im, Re) of e^{-i q.oA}; [4][slots][2 nk].
__global__ void k_grad_table(PeriodicBufs p, int d1, int d2, int slots, double *table) {
    const int id = blockIdx.x * blockDim.x + threadIdx.x, o = id / p.nk, kq = id % p.nk;
    if (o >= slots) return;
    const CellGeom &c = p.cell;
    const double q[3] = {p.kq[3 * kq], p.kq[3 * kq + 1], p.kq[3 * kq + 2]};
    const int n0 = o / (d1 * d2), n1 = o / d2 % d1, n2 = o % d2;
    double t = 0.0;
    for (int e = 0; e < 3; ++e) t += q[e] * (n0 * c.A[e] + n1 * c.A[3 + e] + n2 * c.A[6 + e]);
    double sn, cs;
    sincos(-t, &sn, &cs);
    double *r = table + 2LL * o * p.nk + kq;
    r[0] = cs;
    r[p.nk] = -sn;
    for (int d = 0; d < 3; ++d) {
        double *rd = r + 2LL * (d + 1) * slots * p.nk;
        rd[0] = q[d] * sn;
        rd[p.nk] = q[d] * cs;
    }
}

// Real-space part of the pairs, a warp per pair, lanes over its image offsets; AB [pairs][6][4 slots].
__global__ void __launch_bounds__(256) k_grad_images(AtomBufs b, CellGeom c, double beta, double a, int ntile, int d1, int d2,
                                                     int slots, long long pair0, long long pairs, const double *AB, int ldab,
                                                     double *g_c, double *g_rbar, double *gR, double *gA) {
    const int lane = threadIdx.x & 31;
    double lattice = 0.0;   // of component `lane` < 9
    const long long warps = gridDim.x * 8LL;
    for (long long at = blockIdx.x * 8LL + (threadIdx.x >> 5); at < pairs; at += warps) {
        const Pair p = pair_at(b, ntile, pair0 + at);
        if (!p.valid) continue;
        int lo[3], hi[3];
        image_box(c, p.x, lo, hi);
        double fx[3];
        for (int k = 0; k < 3; ++k) fx[k] = p.x[0] * c.Ainv[k] + p.x[1] * c.Ainv[3 + k] + p.x[2] * c.Ainv[6 + k];
        const double S = b.rbar[p.i] + b.rbar[p.j];
        double s[14];   // zT, zS, zx, zA
#pragma unroll
        for (int t = 0; t < 14; ++t) s[t] = 0.0;
        for (int o = lane; o < slots; o += 32) {
            const int n[3] = {lo[0] + o / (d1 * d2), lo[1] + o / d2 % d1, lo[2] + o % d2};
            if (n[0] > hi[0] || n[1] > hi[1] || n[2] > hi[2]) continue;
            double r[3];
            for (int e = 0; e < 3; ++e) r[e] = p.x[e] + n[0] * c.A[e] + n[1] * c.A[3 + e] + n[2] * c.A[6 + e];
            const double rho2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2];
            if (rho2 >= c.rc * c.rc) continue;
            const double *ab = AB + at * 6 * ldab + o;
            double A[6];
#pragma unroll
            for (int e = 0; e < 6; ++e) A[e] = ab[static_cast<long long>(e) * ldab];
            if (rho2 < 1e-16) {   // the atom itself
                s[0] -= 4.0 * c.gamma * c.gamma * c.gamma / (3.0 * sqrt(kPi)) * (A[0] + A[1] + A[2]);
                continue;
            }
            const double rho = sqrt(rho2), irho = 1.0 / rho;
            const RadialT te = erfc_radial(rho, c.gamma), tb = bare_radial(rho);
            const Fermi g = fermi(rho, S, beta, a);
            const double sr = 1.0 - g.f;
            const double P = te.P - sr * tb.P, W = te.W - sr * tb.W;
            const double dP = te.dP - sr * tb.dP + g.df_drho * tb.P, dW = te.dW - sr * tb.dW + g.df_drho * tb.W;
            const double Ar[3] = {A[0] * r[0] + A[3] * r[1] + A[4] * r[2], A[3] * r[0] + A[1] * r[1] + A[5] * r[2],
                                  A[4] * r[0] + A[5] * r[1] + A[2] * r[2]};
            const double tr = A[0] + A[1] + A[2], rAr = r[0] * Ar[0] + r[1] * Ar[1] + r[2] * Ar[2];
            s[0] += P * tr + W * rAr;
            s[1] += g.df_dS * (tb.P * tr + tb.W * rAr);
            const double rad = (dP * tr + dW * rAr) * irho;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                double B[6];
#pragma unroll
                for (int e = 0; e < 6; ++e) B[e] = ab[static_cast<long long>(e) * ldab + (d + 1) * slots];
                const double rBr = r[0] * (B[0] * r[0] + 2.0 * (B[3] * r[1] + B[4] * r[2])) +
                                   r[1] * (B[1] * r[1] + 2.0 * B[5] * r[2]) + B[2] * r[2] * r[2];
                const double qF = P * (B[0] + B[1] + B[2]) + W * rBr, dF = rad * r[d] + 2.0 * W * Ar[d];
                s[2 + d] += dF + qF;
#pragma unroll
                for (int k = 0; k < 3; ++k) s[5 + 3 * k + d] += n[k] * dF - fx[k] * qF;
            }
        }
#pragma unroll
        for (int t = 0; t < 14; ++t) s[t] = warp_sum(s[t]);
        const double ci = coupling(b, p.i), cj = coupling(b, p.j), cij = ci * cj;
#pragma unroll
        for (int t = 0; t < 9; ++t)
            if (lane == t) lattice += cij * s[5 + t];
        if (lane) continue;
        if (p.i == p.j) {
            atomicAdd(&g_c[p.i], 2.0 * ci * s[0]);
            atomicAdd(&g_rbar[p.i], 2.0 * cij * s[1]);
        } else {
            atomicAdd(&g_c[p.i], cj * s[0]);
            atomicAdd(&g_c[p.j], ci * s[0]);
            atomicAdd(&g_rbar[p.i], cij * s[1]);
            atomicAdd(&g_rbar[p.j], cij * s[1]);
            for (int d = 0; d < 3; ++d) {
                atomicAdd(&gR[3 * p.j + d], cij * s[2 + d]);
                atomicAdd(&gR[3 * p.i + d], -cij * s[2 + d]);
            }
        }
    }
    if (lane < 9) atomicAdd(&gA[lane], lattice);
}

inline int cdiv(long long a, long long b) { return static_cast<int>((a + b - 1) / b); }
inline size_t al(size_t b) { return (b + 255) / 256 * 256; }

// Scratch of the two parts, which follow each other through the same memory: groups of Bloch vectors, and of pairs.
struct Layout {
    int d[3], slots, group, ldn, ldg, ldab;
    long long pairs, chunk;
    size_t left, right, lplanes, rplanes, bytes, out;              // offsets, reciprocal part
    size_t table, tplanes, rows, yplanes, ybytes, ab;              // offsets, real part
    size_t total;
};
constexpr size_t kMostBytes = size_t{8} << 30;
// Groups of vectors and chunks of pairs of lim.cell_sums bytes each.
Layout layout(int N, const CellGeom &c, int nk, int maxG, const ScratchLimits &lim) {
    Layout l{};
    double slots = 1.0;
    for (int k = 0; k < 3; ++k) {
        const double bn = std::sqrt(c.B[3 * k] * c.B[3 * k] + c.B[3 * k + 1] * c.B[3 * k + 1] + c.B[3 * k + 2] * c.B[3 * k + 2]);
        const double d = std::floor(2.0 * (c.rc * bn / (2.0 * kPi) + 1e-9)) + 1.0;
        slots *= d;
        l.d[k] = static_cast<int>(std::min(1e4, d));
    }
    if (slots > 2048.0 || 6.0 * N > 65535.0 || maxG > 65535) return l;   // total 0: not for this cell
    l.slots = l.d[0] * l.d[1] * l.d[2];
    l.ldn = (N + 1) / 2 * 2;
    l.ldg = (maxG + 1) / 2 * 2;
    l.ldab = 4 * l.slots;
    size_t p = 0;
    auto take = [&](size_t n) {
        const size_t at = p;
        p += al(n);
        return at;
    };
    for (l.group = nk;; l.group = (l.group + 1) / 2) {
        p = 0;
        const size_t z = static_cast<size_t>(l.group), n = static_cast<size_t>(N);
        const CrtShape left = crt_shape(6 * N, N, l.group, true, false), right = crt_shape(maxG, N, l.group, true, true);
        l.left = take(8 * z * 12 * n * l.ldn);
        l.right = take(8 * z * 2 * maxG * l.ldn);
        l.lplanes = take(crt_operand_bytes(left));
        l.rplanes = take(crt_operand_bytes(right));
        l.bytes = take(crt_bytes_bytes(6 * N, right.out_rows, l.group));
        l.out = take(8 * z * 12 * n * l.ldg);
        if (p <= lim.cell_sums || l.group == 1) break;
    }
    l.total = p;
    const int ntile = cdiv(N, kQT);
    l.pairs = 256LL * ntile * (ntile + 1) / 2;
    for (l.chunk = l.pairs;; l.chunk = (l.chunk / 2 + 255) / 256 * 256) {
        p = 0;
        const int rows = static_cast<int>(6 * l.chunk);
        l.table = take(8 * static_cast<size_t>(l.ldab) * 2 * nk);
        l.tplanes = take(crt_operand_bytes(crt_shape(l.ldab, 2 * nk, 1, false, true)));
        l.rows = take(8 * static_cast<size_t>(rows) * 2 * nk);
        l.yplanes = take(crt_operand_bytes(crt_shape(rows, 2 * nk, 1, false, false)));
        l.ybytes = take(crt_bytes_bytes(rows, l.ldab, 1));
        l.ab = take(8 * static_cast<size_t>(rows) * l.ldab);
        if (p <= lim.cell_sums || l.chunk == 256) break;
    }
    l.total = std::max(l.total, p);
    if (l.total > kMostBytes) l.total = 0;   // (thousands of atoms, or grids of tens of thousands of vectors)
    return l;
}

}  // namespace

size_t grad_products_bytes(int N, const CellGeom &c, int nk, int maxG, const ScratchLimits &lim) {
    return layout(N, c, nk, maxG, lim).total;
}

cudaError_t grad_products(const AtomBufs &b, const PeriodicBufs &p, double beta, double a, const double *Z, long long ld,
                          double zscale, double *g_c, double *g_rbar, double *gR, double *gA, bool recip, void *work,
                          int *status, cudaStream_t s, const ScratchLimits &lim) {
    const Layout l = layout(b.N, p.cell, p.nk, p.maxG, lim);
    char *w = static_cast<char *>(work);
    auto at = [&](size_t o) { return reinterpret_cast<double *>(w + o); };
    for (int k0 = 0; recip && k0 < p.nk; k0 += l.group) {
        const int g = std::min(l.group, p.nk - k0);
        count_launches(3);
        k_grad_left<<<dim3(cdiv(l.ldn, 64), 6 * b.N, g), 64, 0, s>>>(b, p, Z, ld, zscale, k0, l.ldn, at(l.left));
        k_grad_right<<<dim3(cdiv(l.ldn, 64), p.maxG, g), 64, 0, s>>>(p, b.N, k0, p.maxG, l.ldn, at(l.right));
        const CrtShape left = crt_shape(6 * b.N, b.N, g, true, false), right = crt_shape(p.maxG, b.N, g, true, true);
        const long long lim = 6LL * b.N * l.ldn, rim = static_cast<long long>(p.maxG) * l.ldn, cim = 6LL * b.N * l.ldg;
        const CrtOperand ol = crt_rows(left, at(l.left), at(l.left) + lim, l.ldn, 2 * lim, false, w + l.lplanes, s);
        const CrtOperand orr = crt_rows(right, at(l.right), at(l.right) + rim, l.ldn, 2 * rim, false, w + l.rplanes, s);
        const CrtResult r{1.0, 0.0, nullptr, at(l.out), nullptr, 0, l.ldg, 0, 0, 2 * cim, 0, cim, 0, 0};
        const cudaError_t e = crt_multiply(ol, orr, r, w + l.bytes, status, s);
        if (e != cudaSuccess) return e;
        k_grad_recip<<<dim3(cdiv(b.N, 4), g), 128, 0, s>>>(b, p, k0, at(l.out), l.ldg, g_c, gR, gA);
    }
    const int ntile = cdiv(b.N, kQT);
    count_launches(1);
    k_grad_table<<<cdiv(static_cast<long long>(l.slots) * p.nk, 128), 128, 0, s>>>(p, l.d[1], l.d[2], l.slots, at(l.table));
    const CrtOperand ot = crt_rows(crt_shape(l.ldab, 2 * p.nk, 1, false, true), at(l.table), nullptr, 2 * p.nk, 0, false,
                                   w + l.tplanes, s);
    for (long long p0 = 0; p0 < l.pairs; p0 += l.chunk) {
        const long long n = std::min(l.chunk, l.pairs - p0);
        const int rows = static_cast<int>(6 * n);
        count_launches(2);
        k_grad_rows<<<cdiv(n * p.nk, 256), 256, 0, s>>>(b, p, Z, ld, zscale, ntile, p0, n, at(l.rows));
        const CrtOperand oy = crt_rows(crt_shape(rows, 2 * p.nk, 1, false, false), at(l.rows), nullptr, 2 * p.nk, 0, false,
                                       w + l.yplanes, s);
        const CrtResult r{1.0, 0.0, nullptr, at(l.ab), nullptr, 0, l.ldab, 0, 0, 0, 0, 0, 0, 0};
        const cudaError_t e = crt_multiply(oy, ot, r, w + l.ybytes, status, s);
        if (e != cudaSuccess) return e;
        k_grad_images<<<static_cast<int>(std::min<long long>(cdiv(n, 8), 152 * 8)), 256, 0, s>>>(
            b, p.cell, beta, a, ntile, l.d[1], l.d[2], l.slots, p0, n, at(l.ab), l.ldab, g_c, g_rbar, gR, gA);
    }
    return cudaGetLastError();
}

}  // namespace mbdgb
