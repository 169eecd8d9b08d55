// Q(q) of a cell for every Bloch vector (Eqs. q-matrix, ewald; k_periodic.cu has the formulas) with
// the reciprocal sums as products on the tensor cores and the real-space tensors shared by the
// Bloch vectors.
//
// The reciprocal part of block (i, j) is sum_G w_e(G) conj(S_iG) S_jG for the six components e of the
// symmetric k k^T, w_e = (4 pi/Omega) e^{-k^2/4 gamma^2} k_e k_e' / k^2: for each Bloch vector one
// complex product of 6N x nG by nG x N, formed FP64-accurately by residues (k_crt.cu).  On the FP64 pipe
// (24 operations a pair and G) it took 150 of the 162 ms of the build for 256 atoms, 64 Bloch vectors
// and 1644 vectors G each.  The real-space part is F(r) e^{-i q.r} over images r = x + n A with F real
// and the same for every q: F is tabulated per pair and image offset once (about 150 operations each), and a
// Bloch vector adds F times a phase that depends on the offset alone, times e^{-i q.(x + lo A)} at the end.
// Together 10.2 ms for that cell.  For the FP64 path: the mixed modes round Q further and keep the direct
// build (mbd_api.cu).
#include <algorithm>

#include "cell_pairs.cuh"
#include "internal.h"
#include "pair_math.cuh"

namespace mbdgb {
namespace {

using namespace pairs;
using namespace cellpairs;

// F of one pair at blockIdx.y's image offset (o0, o1, o2) from its first image: T^erfc - (1 - g) T as
// xx, yy, zz, xy, xz, yz, zero beyond the cutoff; F[(offset 6 + e)][pair].
__global__ void __launch_bounds__(256) k_q_images(AtomBufs b, CellGeom c, double beta, double a, int ntile, int d1, int d2,
                                                  double *F, int *status) {
    const Pair p = pair_of(b, ntile);
    const long long pairs = static_cast<long long>(gridDim.x) * 256, id = blockIdx.x * 256LL + threadIdx.x;
    double v[6] = {0, 0, 0, 0, 0, 0};
    if (p.valid) {
        const int o = blockIdx.y, off[3] = {o / (d1 * d2), o / d2 % d1, o % d2};
        int lo[3], hi[3];
        image_box(c, p.x, lo, hi);
        bool in = true;
        for (int e = 0; e < 3; ++e) in = in && lo[e] + off[e] <= hi[e];
        if (in) {
            const int n0 = lo[0] + off[0], n1 = lo[1] + off[1], n2 = lo[2] + off[2];
            double r[3];
            for (int e = 0; e < 3; ++e) r[e] = p.x[e] + n0 * c.A[e] + n1 * c.A[3 + e] + n2 * c.A[6 + e];
            const double rho2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2];
            if (rho2 < 1e-16) {
                if (p.i != p.j || n0 || n1 || n2) atomicOr(status, ST_INPUT);
            } else if (rho2 < c.rc * c.rc) {
                const double rho = sqrt(rho2);
                const RadialT te = erfc_radial(rho, c.gamma), tb = bare_radial(rho);
                const Fermi g = fermi(rho, b.rbar[p.i] + b.rbar[p.j], beta, a);
                const double P = te.P - (1.0 - g.f) * tb.P, W = te.W - (1.0 - g.f) * tb.W;
                v[0] = P + W * r[0] * r[0];
                v[1] = P + W * r[1] * r[1];
                v[2] = P + W * r[2] * r[2];
                v[3] = W * r[0] * r[1];
                v[4] = W * r[0] * r[2];
                v[5] = W * r[1] * r[2];
            }
        }
    }
#pragma unroll
    for (int e = 0; e < 6; ++e) F[(blockIdx.y * 6LL + e) * pairs + id] = v[e];
}

// w_e(G) of Bloch vector k0 + blockIdx.y: [6][ldg], zero beyond its list.
__global__ void k_recip_weights(PeriodicBufs p, int k0, int ldg, double *w) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x, kq = k0 + blockIdx.y;
    if (g >= ldg) return;
    double v[6] = {0, 0, 0, 0, 0, 0};
    if (g < p.gcount[kq]) {
        const double *G = p.G + 3LL * p.glist[static_cast<long long>(kq) * p.maxG + g], *q = p.kq + 3 * kq;
        const double kx = G[0] + q[0], ky = G[1] + q[1], kz = G[2] + q[2], k2 = kx * kx + ky * ky + kz * kz;
        const double c = 4.0 * kPi / p.cell.vol * exp(-k2 * (0.25 / (p.cell.gamma * p.cell.gamma))) / k2;
        v[0] = c * kx * kx;
        v[1] = c * ky * ky;
        v[2] = c * kz * kz;
        v[3] = c * kx * ky;
        v[4] = c * kx * kz;
        v[5] = c * ky * kz;
    }
    for (int e = 0; e < 6; ++e) w[(blockIdx.y * 6LL + e) * ldg + g] = v[e];
}

// The product's operands for Bloch vector k0 + blockIdx.z and atom i = blockIdx.y: rows e N + i of the left
// one, w_e conj(S_i), and row i of the right one, S_i (planar: imaginary parts after the real ones).
__global__ void k_recip_operands(PeriodicBufs p, int N, int k0, int ldg, const double *w, double *left, double *right) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x, i = blockIdx.y, z = blockIdx.z, kq = k0 + z;
    if (g >= ldg) return;
    double2 s = make_double2(0.0, 0.0);
    if (g < p.gcount[kq]) s = p.S[static_cast<long long>(p.glist[static_cast<long long>(kq) * p.maxG + g]) * N + i];
    double *r = right + (z * 2LL * N + i) * ldg + g;
    r[0] = s.x;
    r[static_cast<long long>(N) * ldg] = s.y;
    for (int e = 0; e < 6; ++e) {
        const double we = w[(z * 6LL + e) * ldg + g];
        double *l = left + ((z * 12LL + e) * N + i) * ldg + g;
        l[0] = we * s.x;
        l[6LL * N * ldg] = -we * s.y;
    }
}

// Q of Bloch vector k0 + blockIdx.y from the tabulated images and the reciprocal sums rec[z][2][6 N][ldr].
__global__ void __launch_bounds__(256) k_q_assemble(AtomBufs b, PeriodicBufs p, double *Q, long long ld, int ntile, int k0,
                                                    int d0, int d1, int d2, const double *F, const double *rec, int ldr) {
    extern __shared__ double2 phase[];   // e^{-i q.(o A)} of the image offsets
    const CellGeom &c = p.cell;
    const int z = blockIdx.y, kq = k0 + z, slots = d0 * d1 * d2;
    const double q[3] = {p.kq[3 * kq], p.kq[3 * kq + 1], p.kq[3 * kq + 2]};
    for (int o = threadIdx.x; o < slots; o += 256) {
        const int n0 = o / (d1 * d2), n1 = o / d2 % d1, n2 = o % d2;
        double t = 0.0;
        for (int e = 0; e < 3; ++e) t += q[e] * (n0 * c.A[e] + n1 * c.A[3 + e] + n2 * c.A[6 + e]);
        double sn, cs;
        sincos(-t, &sn, &cs);
        phase[o] = make_double2(cs, sn);
    }
    __syncthreads();
    const Pair pr = pair_of(b, ntile);
    if (!pr.valid) return;
    const int i = pr.i, j = pr.j;
    const long long pairs = static_cast<long long>(gridDim.x) * 256, id = blockIdx.x * 256LL + threadIdx.x;
    double Sr[6] = {0, 0, 0, 0, 0, 0}, Si[6] = {0, 0, 0, 0, 0, 0};
    for (int o = 0; o < slots; ++o) {
        const double2 ph = phase[o];
#pragma unroll
        for (int e = 0; e < 6; ++e) {
            const double f = F[(o * 6LL + e) * pairs + id];
            Sr[e] += f * ph.x;
            Si[e] += f * ph.y;
        }
    }
    int lo[3], hi[3];
    image_box(c, pr.x, lo, hi);
    double t = 0.0;
    for (int e = 0; e < 3; ++e) t += q[e] * (pr.x[e] + lo[0] * c.A[e] + lo[1] * c.A[3 + e] + lo[2] * c.A[6 + e]);
    double sn, cs;
    sincos(-t, &sn, &cs);
    double Tr[6], Ti[6];
    const double *R = rec + z * 12LL * b.N * ldr + static_cast<long long>(i) * ldr + j;
#pragma unroll
    for (int e = 0; e < 6; ++e) {
        Tr[e] = Sr[e] * cs - Si[e] * sn + R[static_cast<long long>(e) * b.N * ldr];
        Ti[e] = Sr[e] * sn + Si[e] * cs + R[(6LL + e) * b.N * ldr];
    }
    if (i == j) {
        const double self = 4.0 * c.gamma * c.gamma * c.gamma / (3.0 * sqrt(kPi));
        for (int e = 0; e < 3; ++e) Tr[e] -= self;
        for (int e = 0; e < 6; ++e) Ti[e] = 0.0;   // (Q is Hermitian with real symmetric diagonal blocks)
    }
    const double pre = b.ombar[i] * b.ombar[j] * sqrt(b.abar0[i] * b.abar0[j]);
    const int ix[9] = {0, 3, 4, 3, 1, 5, 4, 5, 2};
    double *Qr = Q + static_cast<long long>(kq) * 2 * ld * ld, *Qi = Qr + ld * ld;
    const double w2 = b.ombar[i] * b.ombar[i];
    for (int xx = 0; xx < 3; ++xx)
        for (int y = 0; y < 3; ++y) {
            const double vr = pre * Tr[ix[3 * xx + y]] + (i == j && xx == y ? w2 : 0.0);
            const double vi = pre * Ti[ix[3 * xx + y]];
            Qr[(3LL * i + xx) * ld + 3 * j + y] = vr;
            Qi[(3LL * i + xx) * ld + 3 * j + y] = vi;
            if (i != j) {
                Qr[(3LL * j + y) * ld + 3 * i + xx] = vr;
                Qi[(3LL * j + y) * ld + 3 * i + xx] = -vi;
            }
        }
}

inline int cdiv(long long a, long long b) { return static_cast<int>((a + b - 1) / b); }
inline size_t al(size_t b) { return (b + 255) / 256 * 256; }

// Scratch: the image table, and for a group of Bloch vectors the product's arrays.
struct Layout {
    int d[3], slots, group, ldg, ldr;
    CrtShape left, right;
    size_t images, weights, lrows, rrows, lplanes, rplanes, bytes, rec, total;   // offsets
};
constexpr size_t kImageBytes = size_t{512} << 20;  // of the image table at most
// Groups of lim.cell_sums bytes of the product's arrays: 4 Bloch vectors of the 256-atom cell, nine times the chip in tiles.
Layout layout(int N, const CellGeom &c, int nk, int maxG, const ScratchLimits &lim) {
    Layout l{};
    l.slots = 1;
    double slots = 1.0;
    for (int k = 0; k < 3; ++k) {
        const double bn = std::sqrt(c.B[3 * k] * c.B[3 * k] + c.B[3 * k + 1] * c.B[3 * k + 1] + c.B[3 * k + 2] * c.B[3 * k + 2]);
        slots *= std::floor(2.0 * (c.rc * bn / (2.0 * kPi) + 1e-9)) + 1.0;
        l.d[k] = static_cast<int>(std::min(1e4, std::floor(2.0 * (c.rc * bn / (2.0 * kPi) + 1e-9)) + 1.0));
    }
    const int ntile = cdiv(N, kQT);
    const double pairs = 256.0 * ntile * (ntile + 1) / 2;
    if (slots > 2048.0 || slots * 48.0 * pairs > static_cast<double>(kImageBytes)) return l;   // total 0: not for this cell
    l.slots = l.d[0] * l.d[1] * l.d[2];
    l.ldg = static_cast<int>((maxG + 1) / 2 * 2);
    l.ldr = (N + 1) / 2 * 2;
    for (l.group = nk;; l.group = (l.group + 1) / 2) {
        l.left = crt_shape(6 * N, maxG, l.group, true, false);
        l.right = crt_shape(N, maxG, l.group, true, true);
        size_t p = 0;
        auto take = [&](size_t n) {
            const size_t at = p;
            p += al(n);
            return at;
        };
        const size_t z = static_cast<size_t>(l.group), n = static_cast<size_t>(N);
        l.weights = take(8 * z * 6 * l.ldg);
        l.lrows = take(8 * z * 12 * n * l.ldg);
        l.rrows = take(8 * z * 2 * n * l.ldg);
        l.lplanes = take(crt_operand_bytes(l.left));
        l.rplanes = take(crt_operand_bytes(l.right));
        l.bytes = take(crt_bytes_bytes(6 * N, l.right.out_rows, l.group));
        l.rec = take(8 * z * 12 * n * l.ldr);
        if (p <= lim.cell_sums || l.group == 1) {
            l.images = p;
            l.total = p + al(static_cast<size_t>(48.0 * pairs) * l.slots);
            return l;
        }
    }
}

}  // namespace

size_t build_q_products_bytes(int N, const CellGeom &c, int nk, int maxG, const ScratchLimits &lim) {
    return layout(N, c, nk, maxG, lim).total;
}

cudaError_t build_q_products(const AtomBufs &b, const PeriodicBufs &p, double beta, double a, double *Q, long long ld,
                             void *work, int *status, cudaStream_t s, const ScratchLimits &lim) {
    const Layout l = layout(b.N, p.cell, p.nk, p.maxG, lim);
    char *w = static_cast<char *>(work);
    auto at = [&](size_t o) { return reinterpret_cast<double *>(w + o); };
    const int ntile = cdiv(b.N, kQT), tiles = ntile * (ntile + 1) / 2;
    count_launches(1);
    k_q_images<<<dim3(tiles, l.slots), 256, 0, s>>>(b, p.cell, beta, a, ntile, l.d[1], l.d[2], at(l.images), status);
    for (int k0 = 0; k0 < p.nk; k0 += l.group) {
        const int g = std::min(l.group, p.nk - k0);
        count_launches(3);
        k_recip_weights<<<dim3(cdiv(l.ldg, 128), g), 128, 0, s>>>(p, k0, l.ldg, at(l.weights));
        k_recip_operands<<<dim3(cdiv(l.ldg, 128), b.N, g), 128, 0, s>>>(p, b.N, k0, l.ldg, at(l.weights), at(l.lrows),
                                                                       at(l.rrows));
        const CrtShape left = crt_shape(6 * b.N, p.maxG, g, true, false), right = crt_shape(b.N, p.maxG, g, true, true);
        const long long lim = 6LL * b.N * l.ldg, rim = static_cast<long long>(b.N) * l.ldg, cim = 6LL * b.N * l.ldr;
        const CrtOperand ol = crt_rows(left, at(l.lrows), at(l.lrows) + lim, l.ldg, 2 * lim, false, w + l.lplanes, s);
        const CrtOperand orr = crt_rows(right, at(l.rrows), at(l.rrows) + rim, l.ldg, 2 * rim, false, w + l.rplanes, s);
        const CrtResult r{1.0, 0.0, nullptr, at(l.rec), nullptr, 0, l.ldr, 0, 0, 2 * cim, 0, cim, 0, 0};
        const cudaError_t e = crt_multiply(ol, orr, r, w + l.bytes, status, s);
        if (e != cudaSuccess) return e;
        k_q_assemble<<<dim3(tiles, g), 256, sizeof(double2) * l.slots, s>>>(b, p, Q, ld, ntile, k0, l.d[0], l.d[1], l.d[2],
                                                                           at(l.images), at(l.rec), l.ldr);
    }
    return cudaGetLastError();
}

}  // namespace mbdgb
