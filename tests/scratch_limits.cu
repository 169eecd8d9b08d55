// C entry points to the limits of the scratch of the tensor-core products, for the GPU tests.  Test
// infrastructure: built by tests/test_gpu_scratch_limits.py and linked to the library.
#include "internal.h"

using namespace mbdgb;

namespace {
ScratchLimits limits(int none, int panel, size_t trailing, int strip, size_t cell_products, size_t cell_sums) {
    ScratchLimits l;
    l.none = none != 0;
    l.panel = panel;
    l.trailing = trailing;
    l.strip = strip;
    l.cell_products = cell_products;
    l.cell_sums = cell_sums;
    return l;
}
}  // namespace

extern "C" void limit_context(void *ctx, int none, int panel, size_t trailing, int strip, size_t cell_products,
                              size_t cell_sums) {
    set_scratch_limits(static_cast<mbd_ctx *>(ctx), limits(none, panel, trailing, strip, cell_products, cell_sums));
}

// The factorisation with a trailing product of at most `trailing` bytes, in strips of at least `strip` columns.
extern "C" size_t limited_cholesky_bytes(long long ld, int batch, size_t trailing, int strip) {
    return cholesky_crt_bytes(ld, batch, limits(0, 8192, trailing, strip, 0, 0));
}
extern "C" int limited_cholesky(double *A, long long ld, int batch, double *dinv, void *work, int *status, size_t trailing,
                                int strip) {
    return static_cast<int>(cholesky_crt(A, ld, ld * ld, batch, dinv, work, status, nullptr,
                                         limits(0, 8192, trailing, strip, 0, 0)));
}
