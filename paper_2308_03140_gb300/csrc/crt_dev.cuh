// Device pieces of the residue products shared by k_crt.cu and the Cholesky factorisation
// (k_chol.cu).
#pragma once
#include <math_constants.h>

#include "crt64.cuh"

namespace mbdgb {
namespace crt {

// v 2^-(ea + eb): the exponent field directly while the result stays a normal number.
__device__ __forceinline__ double scaled_down(double v, int ea, int eb) {
    if (ea == kBadRow || eb == kBadRow) return CUDART_NAN;
    const int e = ea + eb, hi = __double2hiint(v), f = (hi >> 20) & 0x7ff, to = f - e;
    if (f > 0 && f < 2047 && to > 0 && to < 2047) return __hiloint2double(hi - (e << 20), __double2loint(v));
    return v == 0.0 ? v : scalbn(v, -e);
}

}  // namespace crt
}  // namespace mbdgb
