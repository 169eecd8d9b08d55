// Pairs of a cell's atoms by tiles, and their lattice images (k_periodic.cu, k_qbuild.cu, k_qgrad.cu).
#pragma once
#include "internal.h"
#include "pair_math.cuh"

namespace mbdgb {
namespace cellpairs {

using pairs::kPi;

constexpr int kQT = 16;   // atom tile edge: 16 x 16 threads, tile pairs I <= J

__device__ __forceinline__ void tile_pair(int t, int ntile, int &I, int &J) {
    I = 0;
    while (t >= ntile - I) { t -= ntile - I; ++I; }
    J = I + t;
}

__device__ __forceinline__ double frac_coord(const CellGeom &c, const double *v, int k) {
    return v[0] * c.Ainv[k] + v[1] * c.Ainv[3 + k] + v[2] * c.Ainv[6 + k];
}

// First and last image index of each direction for separation x: r = x + n A within the cutoff needs
// n_c in [-L_c - f_c, L_c - f_c] (f = fractional x, L_c = rc |b_c| / 2 pi).
__device__ __forceinline__ void image_box(const CellGeom &c, const double *x, int *lo, int *hi) {
    for (int k = 0; k < 3; ++k) {
        const double bn = sqrt(c.B[3 * k] * c.B[3 * k] + c.B[3 * k + 1] * c.B[3 * k + 1] + c.B[3 * k + 2] * c.B[3 * k + 2]);
        const double L = c.rc * bn / (2.0 * kPi) + 1e-9, f = frac_coord(c, x, k);
        lo[k] = static_cast<int>(ceil(-L - f));
        hi[k] = static_cast<int>(floor(L - f));
    }
}

struct Pair {
    int i, j;
    bool valid;
    double x[3];
};
__device__ __forceinline__ Pair pair_of(const AtomBufs &b, int ntile) {
    int I, J;
    tile_pair(blockIdx.x, ntile, I, J);
    const int ty = threadIdx.x / kQT, tx = threadIdx.x % kQT;
    Pair p;
    p.i = I * kQT + ty;
    p.j = J * kQT + tx;
    p.valid = p.i < b.N && p.j < b.N && (I < J || ty <= tx);
    for (int e = 0; e < 3; ++e) p.x[e] = p.valid ? b.R[3 * p.j + e] - b.R[3 * p.i + e] : 0.0;
    return p;
}

}  // namespace cellpairs
}  // namespace mbdgb
