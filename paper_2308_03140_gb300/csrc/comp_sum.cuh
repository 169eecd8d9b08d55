// Compensated FP64 sums (error-free additions) of a thread, a warp and a block.
#pragma once
#include <cuda_runtime.h>

namespace mbdgb {
namespace comp {

__device__ __forceinline__ void two_sum(double a, double b, double &s, double &e) {
    s = a + b;
    const double bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// A running sum s and the sum c of what its additions lost.
struct Sum {
    double s = 0.0, c = 0.0;
    __device__ __forceinline__ void add(double x) {
        double t, e;
        two_sum(s, x, t, e);
        s = t;
        c += e;
    }
    __device__ __forceinline__ void add(const Sum &o) {
        add(o.s);
        c += o.c;
    }
    __device__ __forceinline__ double value() const { return s + c; }
};

// Sum over the block (256 threads), the same in every thread; sh: 8 pairs of shared memory.  A tree of 8 levels: one thread adding up 256 partial sums took 30 to 80 us, which is as long as the
// products of a small system.
__device__ __forceinline__ Sum block_sum256(Sum v, double (*sh)[2]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto fold = [&](int o) {
        Sum w;
        w.s = __shfl_xor_sync(0xffffffffu, v.s, o);
        w.c = __shfl_xor_sync(0xffffffffu, v.c, o);
        v.add(w);
    };
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) fold(o);
    if (lane == 0) {
        sh[warp][0] = v.s;
        sh[warp][1] = v.c;
    }
    __syncthreads();
    v.s = sh[lane & 7][0];
    v.c = sh[lane & 7][1];
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) fold(o);
    __syncthreads();
    return v;
}

}  // namespace comp
}  // namespace mbdgb
