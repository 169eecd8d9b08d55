// Batched triangular solves with 3 right-hand sides for the screening systems of
// Eq. (scs): L y = b, then L^T x = y, with L from the blocked Cholesky factorisations
// (FP64 or FP32) and the inverses of its 64x64 diagonal blocks.
//
// Block-column form, one launch per diagonal block I and direction: with the solution x_I of
// block I known, every CTA subtracts the block's contribution from its own slice of the rows still to be
// solved, and the CTA whose slice is the next block then solves that block's 64x3 system (a triangular
// product with the stored inverse) and stores its solution for the next launch.  The chain of
// launches bounds it, so a launch does little before its first dependent load: launches overlap
// (programmatic dependent launch) and each loads its slice of L, and the next block's inverse, before it waits
// for the one before.  With every CTA solving block I for itself a launch took 15.7 (forward) and
// 10.2 us (backward) on average at order 6016 (16 FP32 matrices), 8.9 and 7.8 so, and less where they overlap.
//
// Forward:  y_I = D_I^{-1} b_I;  b_J -= L_JI y_I  (J > I; CTA slice = 64 rows of L, four
//           threads per row),
//           b (the caller's array) is the running right-hand side, y goes to work.
// Backward: x_I = D_I^{-T} y_I;  y_J -= L_IJ^T x_I (J < I; CTA slice = 64 columns),
//           work is the running right-hand side, x goes to the caller's array.
// No launch both reads and writes one block of one array: block I of the output array is read, block I +- 1
// of it written, and blocks of the running right-hand side updated by their own CTAs only.
#include "internal.h"

namespace mbdgb {
namespace {

// Everything before this may run while the launch before is still running; what that one wrote may be
// read only after it.
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

// The 64x64 inverse of a diagonal block into shared memory (256 threads, coalesced).
template <typename T>
__device__ __forceinline__ void load_inverse(const T *Di, T (*D)[65]) {
#pragma unroll
    for (int e = threadIdx.x; e < 64 * 64; e += 256) D[e >> 6][e & 63] = Di[e];
}
// out [64][3] = D^{-1} s (forward) or D^{-T} s (backward) from the inverse in shared memory.
template <typename T, bool BWD>
__device__ __forceinline__ void diag_solve(const T (*D)[65], const T (*s)[3], T *out) {
    const int t = threadIdx.x;
    if (t >= 192) return;
    const int r = t / 3, c = t % 3;
    T v = 0;
#pragma unroll 16
    for (int k = 0; k < 64; ++k) {
        const T d = BWD ? D[k][r] : D[r][k];
        if (BWD ? k >= r : k <= r) v += d * s[k][c];
    }
    out[t] = v;
}

// First block: y_0 = D_0^{-1} b_0, or x_last = D_last^{-T} y_last.
template <typename T, bool BWD>
__global__ void __launch_bounds__(256) k_trsv_first(const T *dinv, long long dstride, const T *rhs, T *out,
                                                    long long xstride, int I) {
    __shared__ T D[64][65], s[64][3];
    const long long b = blockIdx.x;
    let_next_start();
    load_inverse(dinv + b * dstride + static_cast<long long>(I) * 4096, D);
    wait_for_previous();
    if (threadIdx.x < 192) s[threadIdx.x / 3][threadIdx.x % 3] = rhs[b * xstride + 192LL * I + threadIdx.x];
    __syncthreads();
    diag_solve<T, BWD>(D, s, out + b * xstride + 192LL * I);
}

// kWide: L in 16-byte loads, for an L that starts on 16 bytes (its rows are multiples of 64 entries); callers may
// also pass one that does not, which is read entry by entry.
template <typename T, bool kWide>
__global__ void __launch_bounds__(256) k_trsv_fwd_block(const T *L, long long ld, long long mstride, const T *dinv,
                                                        long long dstride, T *X, T *W, long long xstride, int I) {
    const long long b = blockIdx.x;   // (the batch first: the CTAs of the next blocks start first)
    const T *Lb = L + b * mstride;
    T *Xb = X + b * xstride, *Wb = W + b * xstride;
    __shared__ T D[64][65], s[64][3], x[64][3];
    const long long I0 = static_cast<long long>(I) * 64;
    const bool next = blockIdx.y == 0;   // this CTA's rows are block I + 1
    let_next_start();
    // rows of this CTA: 64 rows starting after block I; four threads per row, each taking
    // 16 consecutive columns of the block, combined by two shuffles
    const long long r0 = I0 + 64 + static_cast<long long>(blockIdx.y) * 64;
    const int rr = threadIdx.x >> 2, q = threadIdx.x & 3;
    const T *Lq = Lb + (r0 + rr) * ld + I0 + 16 * q;
    alignas(16) T l[16];
#pragma unroll
    for (int c = 0; c < 16; c += kWide ? 16 / sizeof(T) : 1) {
        if constexpr (kWide) *reinterpret_cast<int4 *>(l + c) = *reinterpret_cast<const int4 *>(Lq + c);
        else l[c] = Lq[c];
    }
    if (next) load_inverse(dinv + b * dstride + static_cast<long long>(I + 1) * 4096, D);
    wait_for_previous();
    if (threadIdx.x < 192) x[threadIdx.x / 3][threadIdx.x % 3] = Wb[3 * I0 + threadIdx.x];
    __syncthreads();
    T a0 = 0, a1 = 0, a2 = 0;
#pragma unroll
    for (int c = 0; c < 16; ++c) {
        a0 += l[c] * x[16 * q + c][0];
        a1 += l[c] * x[16 * q + c][1];
        a2 += l[c] * x[16 * q + c][2];
    }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        a0 += __shfl_xor_sync(0xffffffffu, a0, o);
        a1 += __shfl_xor_sync(0xffffffffu, a1, o);
        a2 += __shfl_xor_sync(0xffffffffu, a2, o);
    }
    if (q == 0) {
        T *xq = Xb + 3 * (r0 + rr);
        const T b0 = xq[0] - a0, b1 = xq[1] - a1, b2 = xq[2] - a2;
        if (next) {
            s[rr][0] = b0;
            s[rr][1] = b1;
            s[rr][2] = b2;
        } else {
            xq[0] = b0;
            xq[1] = b1;
            xq[2] = b2;
        }
    }
    if (!next) return;
    __syncthreads();
    diag_solve<T, false>(D, s, Wb + 3 * (I0 + 64));
}

template <typename T>
__global__ void __launch_bounds__(256) k_trsv_bwd_block(const T *L, long long ld, long long mstride, const T *dinv,
                                                        long long dstride, T *X, T *W, long long xstride, int I) {
    const long long b = blockIdx.x;
    const T *Lb = L + b * mstride;
    T *Xb = X + b * xstride, *Wb = W + b * xstride;
    __shared__ T D[64][65], s[64][3], x[64][3];
    __shared__ T part[4][64][3];
    const long long I0 = static_cast<long long>(I) * 64;
    const bool next = blockIdx.y == 0;   // this CTA's columns are block I - 1
    let_next_start();
    // columns of this CTA: 64 columns j < I0, counted from block I - 1 down
    const long long c0 = I0 - 64 - static_cast<long long>(blockIdx.y) * 64;
    const int t = threadIdx.x, col = t & 63, grp = t >> 6;
    T l[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) l[k] = Lb[(I0 + grp + 4 * k) * ld + c0 + col];   // rows of block I
    if (next) load_inverse(dinv + b * dstride + static_cast<long long>(I - 1) * 4096, D);
    wait_for_previous();
    if (t < 192) x[t / 3][t % 3] = Xb[3 * I0 + t];
    __syncthreads();
    T a0 = 0, a1 = 0, a2 = 0;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const int i = grp + 4 * k;
        a0 += l[k] * x[i][0];
        a1 += l[k] * x[i][1];
        a2 += l[k] * x[i][2];
    }
    part[grp][col][0] = a0; part[grp][col][1] = a1; part[grp][col][2] = a2;
    __syncthreads();
    if (t < 192) {
        const int cc = t / 3, k = t % 3;
        T *w = Wb + 3 * (c0 + cc) + k;
        const T v = *w - (part[0][cc][k] + part[1][cc][k] + part[2][cc][k] + part[3][cc][k]);
        if (next) s[cc][k] = v;
        else *w = v;
    }
    if (!next) return;
    __syncthreads();
    diag_solve<T, true>(D, s, Xb + 3 * (I0 - 64));
}

}  // namespace

template <typename T>
void trsv_blocked(const T *L, long long ld, long long mstride, int batch, const T *dinv, T *X, T *W, long long xstride,
                  cudaStream_t s) {
    const int nb = static_cast<int>(ld / 64);
    const long long dstride = static_cast<long long>(nb) * 4096;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cfg.attrs = attr;
    // The first launch of a direction starts only after what came before: a kernel that is not part of this
    // chain need not have finished its writes of L when it lets the next one start.
    cfg.numAttrs = 0;
    cfg.gridDim = dim3(batch);
    count_launches(2 * nb);
    cudaLaunchKernelEx(&cfg, k_trsv_first<T, false>, dinv, dstride, static_cast<const T *>(X), W, xstride, 0);
    cfg.numAttrs = 1;
    const bool wide = (reinterpret_cast<uintptr_t>(L) & 15) == 0 && mstride * sizeof(T) % 16 == 0;
    for (int I = 0; I + 1 < nb; ++I) {
        cfg.gridDim = dim3(batch, nb - 1 - I);   // 64-row slices below block I
        if (wide) cudaLaunchKernelEx(&cfg, k_trsv_fwd_block<T, true>, L, ld, mstride, dinv, dstride, X, W, xstride, I);
        else cudaLaunchKernelEx(&cfg, k_trsv_fwd_block<T, false>, L, ld, mstride, dinv, dstride, X, W, xstride, I);
    }
    cfg.gridDim = dim3(batch);
    cudaLaunchKernelEx(&cfg, k_trsv_first<T, true>, dinv, dstride, static_cast<const T *>(W), X, xstride, nb - 1);
    for (int I = nb - 1; I > 0; --I) {
        cfg.gridDim = dim3(batch, I);            // 64-column slices left of block I
        cudaLaunchKernelEx(&cfg, k_trsv_bwd_block<T>, L, ld, mstride, dinv, dstride, X, W, xstride, I);
    }
}

template void trsv_blocked<double>(const double *, long long, long long, int, const double *, double *, double *,
                                   long long, cudaStream_t);
template void trsv_blocked<float>(const float *, long long, long long, int, const float *, float *, float *,
                                  long long, cudaStream_t);

}  // namespace mbdgb
