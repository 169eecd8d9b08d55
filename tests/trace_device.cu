// C entry point to the block traces of the mixed modes' correction (csrc/k_tc.cu), for the GPU tests.  Test
// infrastructure: built by tests/test_gpu_block_trace.py and linked to the library.
#include "internal.h"

extern "C" void block_traces(const double *V, const double *W, long long ld, int N, double sqrt_s, double *tq) {
    mbdgb::block_trace_sqrt(V, W, ld, N, sqrt_s, tq, nullptr);
}
