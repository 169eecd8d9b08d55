// FP64-accurate products C = alpha A op(B) + beta D on the bf16 tensor cores (crt64.cuh).
//
// FP64 runs at about 1.05 TFLOP/s on this part, bf16 at 1900: an FP64 product is 15 bf16 products
// of residues, whose sums are exact, and two passes over memory.  Three kernels:
//   k_crt_rows    rows of an FP64 operand -> their exponents and 15 planes of bf16 residues, K-major
//   k_crt_gemm    the products of the planes, each reduced by its modulus to one byte per entry
//   k_crt_result  bytes -> FP64, with alpha, beta D, and the mirrored or transposed copies
#include <algorithm>
#include <atomic>

#include <cuda.h>
#include <cudaTypedefs.h>

#include "crt_dev.cuh"
#include "internal.h"
#include "tc_ops.cuh"

namespace mbdgb {
namespace {

using namespace tcops;
using crt::kMod;

// ---- operands -------------------------------------------------------------------------------
// kThreads threads take one row: its 2-norm, then four consecutive entries at a time to limbs and
// 15 residues, stored as bf16 (an integer of at most 8 bits is the upper half of its FP32 word).
// A complex operand's row is [re | im] (the left operand) or gives the two rows [re | -im] and
// [im | re] (the right one, whose rows are the columns of B; conj takes them from a Hermitian B's
// own rows), so that the complex product is the real one
//   [Ar | Ai] [[Br | -Bi], [Bi | Br]]^T = [Re C | Im C].
// Bound by HBM for long rows: 8 bytes in (the second read of a row comes from L2), 30 out.
struct RowsArgs {
    const double *re, *im;   // im: complex operands (else null)
    long long ld, stride;    // row pitch; batch items stride apart
    int rows, K;
    int right, conj;         // complex: the right operand's two rows per column
    int half, second;        // entries from one half row to the next; output rows to the second set
    __nv_bfloat16 *planes;   // [batch][kMod][out_rows][pitch]
    long long pitch, plane, item;   // entries: row, plane, batch item
    int *exps;               // [batch][out_rows]
    int out_rows;
};

template <int kThreads>
__device__ __forceinline__ double row_sum(double v, double *sh, int t) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (kThreads == 32) return v;
    if ((t & 31) == 0) sh[t >> 5] = v;
    __syncthreads();
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) s += sh[w];
    __syncthreads();
    return s;
}
template <int kThreads>
__device__ __forceinline__ double row_max(double v, double *sh, int t) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (kThreads == 32) return v;
    if ((t & 31) == 0) sh[t >> 5] = v;
    __syncthreads();
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) s = fmax(s, sh[w]);
    __syncthreads();
    return s;
}

__device__ __forceinline__ void load4(const double *row, int k, int K, double (&v)[4]) {
    if (k + 4 <= K) {
        const double2 a = *reinterpret_cast<const double2 *>(row + k), b = *reinterpret_cast<const double2 *>(row + k + 2);
        v[0] = a.x;
        v[1] = a.y;
        v[2] = b.x;
        v[3] = b.y;
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = k + j < K ? row[k + j] : 0.0;
    }
}

__device__ __forceinline__ void fit(double (&v)[4], bool bad, double rest) {
    if (!bad && rest == 1.0) return;
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = bad ? 0.0 : v[j] * rest;
}

// Residues of four entries into the planes at `out` (and negated at `neg`, or the same at `same`).
__device__ __forceinline__ void put4(const double (&v)[4], double scale, long long plane, __nv_bfloat16 *out,
                                     __nv_bfloat16 *neg, __nv_bfloat16 *same) {
    crt::Limbs l[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) l[j] = crt::limbs(__double2ll_rn(v[j] * scale));
    crt::each_modulus([&](auto I) {
        uint32_t f[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) f[j] = __float_as_uint(crt::residue<decltype(I)::value>(l[j]));
        const uint2 w = make_uint2(__byte_perm(f[0], f[1], 0x7632), __byte_perm(f[2], f[3], 0x7632));
        const long long o = decltype(I)::value * plane;
        *reinterpret_cast<uint2 *>(out + o) = w;
        if (neg) *reinterpret_cast<uint2 *>(neg + o) = make_uint2(w.x ^ 0x80008000u, w.y ^ 0x80008000u);
        if (same) *reinterpret_cast<uint2 *>(same + o) = w;
    });
}

template <int kThreads>
__global__ void __launch_bounds__(128) k_crt_rows(RowsArgs g) {
    constexpr int kRows = 128 / kThreads;
    __shared__ double sh[4];
    const int r = blockIdx.x * kRows + threadIdx.x / kThreads, t = threadIdx.x % kThreads;
    if (r >= g.rows) return;   // whole warps: a row is a warp's or the block's
    const long long b = blockIdx.y;
    const double *re = g.re + b * g.stride + r * g.ld, *im = g.im ? g.im + b * g.stride + r * g.ld : nullptr;
    double ss = 0.0;
    for (int k = 4 * t; k < g.K; k += 4 * kThreads) {
        double v[4];
        load4(re, k, g.K, v);
        ss += v[0] * v[0] + v[1] * v[1] + v[2] * v[2] + v[3] * v[3];
        if (im) {
            load4(im, k, g.K, v);
            ss += v[0] * v[0] + v[1] * v[1] + v[2] * v[2] + v[3] * v[3];
        }
    }
    ss = row_sum<kThreads>(ss, sh, t);
    int e;
    if (ss > 1e-280 && ss < 1e280) {
        e = crt::row_exponent(sqrt(ss));
    } else {   // squares out of range (or a zero row): the norm from the scaled row
        double mx = 0.0;
        for (int k = t; k < g.K; k += kThreads) {   // (a NaN counts as infinite)
            const double a = fabs(re[k]), c = im ? fabs(im[k]) : 0.0;
            mx = fmax(mx, a <= crt::kMaxDouble && c <= crt::kMaxDouble ? fmax(a, c) : CUDART_INF);
        }
        mx = row_max<kThreads>(mx, sh, t);
        if (mx == 0.0 || mx > crt::kMaxDouble) {
            e = crt::row_exponent(mx);
        } else {
            int x;
            frexp(mx, &x);
            double s2 = 0.0;
            for (int k = t; k < g.K; k += kThreads) {
                const double a = ldexp(re[k], -x), c = im ? ldexp(im[k], -x) : 0.0;
                s2 += a * a + c * c;
            }
            e = crt::row_exponent(sqrt(row_sum<kThreads>(s2, sh, t)));   // of the row times 2^-x
            e -= x;
        }
    }
    if (t == 0) {
        int *eo = g.exps + b * g.out_rows + r;
        eo[0] = e;
        if (g.right && im) eo[g.second] = e;
    }
    const bool bad = e == crt::kBadRow;   // its residues are zeros; its products are NaN
    const double scale = bad ? 0.0 : crt::pow2(min(e, 1000));
    const double rest = e > 1000 && !bad ? crt::pow2(e - 1000) : 1.0;   // rows below 1e-283 are scaled twice
    __nv_bfloat16 *out = g.planes + b * g.item + r * g.pitch;
    for (int k = 4 * t; k < g.half; k += 4 * kThreads) {   // entries K .. half - 1 are zeros
        double v[4];
        load4(re, k, g.K, v);
        fit(v, bad, rest);
        __nv_bfloat16 *o2 = im && g.right ? out + g.second * g.pitch : nullptr;
        put4(v, scale, g.plane, out + k, nullptr, o2 ? o2 + g.half + k : nullptr);
        if (!im) continue;
        load4(im, k, g.K, v);
        fit(v, bad, rest);
        if (!g.right) {
            put4(v, scale, g.plane, out + g.half + k, nullptr, nullptr);
        } else if (!g.conj) {   // [re | -im], [im | re]
            put4(v, scale, g.plane, o2 + k, out + g.half + k, nullptr);
        } else {
            put4(v, scale, g.plane, out + g.half + k, o2 + k, nullptr);
        }
    }
}

// ---- products -------------------------------------------------------------------------------
// Work item: (batch item, modulus, tile of 256 x kN entries).  The wide form, kN = 256:  a cluster of two CTAs computes it
// with tcgen05.mma.cta_group::2 (M = 256, N = 256): CTA r stages rows 128 r .. 128 r + 127 of A's and of B's
// 256 (32 KB per stage of 64 entries, six stages), so the two together load 64 KB for 512 cycles of
// MMA, and holds rows 128 r .. of the tile in its tensor memory, in two buffers of 256 columns.
// A single CTA on 128 x 256 tiles would load 48 KB in the same time, more than an SM takes in.
// Every 1024 products the eight epilogue warps reduce the buffer (exact integers) by the modulus and
// add it to their 128 sums a thread, four FP32 operations an entry, while the other buffer fills.
// The TMA and MMA warps run uniformly and issue from an elected lane: from a branch on the lane each MMA
// took about 200 cycles to issue, more than its 128 to run (a whole product of order 6016 with its
// conversions: 6.98 ms, 4.54 so, 4.30 with sums of 1024 products instead of 512; order 3000 1.06, then
// 0.92, 0.90, and 0.71 with rows on 128-byte lines).  The MMAs alone run for 2.76 ms of the 3.3 ms of this
// kernel at order 6016, the loads alone for 3.0 (17 TB/s out of L2), which bound it.
// Clusters are persistent and walk the items in order, so that those in flight share a modulus and
// neighbouring tiles in L2.  Barriers as in the CTA-pair GEMM (k_tc.cu): full, cfree on the even CTA; empty,
// cfull, done in both.  Every wait is bounded; on a timeout the kernel raises ST_TC_TIMEOUT,
// waits (bounded) for its copies and MMAs, frees its tensor memory and returns.
// Narrow tiles (256 x 64) serve the Cholesky factorisation's 64-column blocks and small matrices.
constexpr int kTileM = 256;
constexpr int kHalfBytes = 128 * 128;              // 128 rows of 64 bf16
template <int kN>
struct Tile {
    static constexpr int kStageBytes = kHalfBytes + kN / 2 * 128;   // per CTA
    static constexpr int kStages = kN == 256 ? 6 : 8;
    static constexpr int kSmem = kStages * kStageBytes + 1024 + 256;
};
constexpr int kWarps = 10;                         // 8 epilogue, TMA, MMA

__constant__ float c_m[kMod] = {256, 255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197};
__constant__ float c_back[kMod] = {
    crt::inverse_of_rest(0),  crt::inverse_of_rest(1),  crt::inverse_of_rest(2),  crt::inverse_of_rest(3),
    crt::inverse_of_rest(4),  crt::inverse_of_rest(5),  crt::inverse_of_rest(6),  crt::inverse_of_rest(7),
    crt::inverse_of_rest(8),  crt::inverse_of_rest(9),  crt::inverse_of_rest(10), crt::inverse_of_rest(11),
    crt::inverse_of_rest(12), crt::inverse_of_rest(13), crt::inverse_of_rest(14)};

struct GemmCrt {
    int M, N, K;             // K: entries of a plane's row (a multiple of 8; the tail reads as zeros)
    int batch, tiles_m, tiles_n, tiles;
    int half;                // 1: tiles on or above the diagonal only, 2: on or below it
    uint8_t *Y;              // [batch][kMod][M][ldy]
    long long ldy;
    int *err;
};

__device__ __forceinline__ void tma_load_3d_pair(void *dst, const CUtensorMap *map, int x, int y, int z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];\n" ::"r"(
            su32(dst)),
        "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}
// bf16 operands, FP32 accumulator, both K-major, M = 256 (two CTAs), N = kN.
template <int kN>
__device__ __forceinline__ void mma_pair(uint32_t tmem, uint64_t a, uint64_t b, uint32_t acc) {
    constexpr uint32_t id = (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(kN >> 3) << 17) |
                            (static_cast<uint32_t>(kTileM >> 4) << 24);
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(a), "l"(b), "r"(id), "r"(acc));
}
// Arrival on the barrier at this shared-memory address in both CTAs of the pair, once the MMAs so far
// are done.
__device__ __forceinline__ void commit_both(uint32_t addr) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n" ::"r"(addr),
        "h"(static_cast<unsigned short>(3))
        : "memory");
}

// Tile t of the walk: columns of tiles in groups of eight rows, or the triangle's columns (rows).
__device__ __forceinline__ void crt_tile(const GemmCrt &g, int t, int &tm, int &tn) {
    if (g.half) {
        int c = static_cast<int>((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);
        while ((c + 1) * (c + 2) / 2 <= t) ++c;
        while (c * (c + 1) / 2 > t) --c;
        const int r = t - c * (c + 1) / 2;   // r <= c
        tm = g.half == 1 ? r : c;
        tn = g.half == 1 ? c : r;
        return;
    }
    const int group = t / (8 * g.tiles_n), first = group * 8, rows = min(8, g.tiles_m - first);
    const int l = t - group * 8 * g.tiles_n;
    tm = first + l % rows;
    tn = l / rows;
}

template <int kN>
__global__ void __launch_bounds__(32 * kWarps, 1)
    k_crt_gemm(const __grid_constant__ CUtensorMap mA, const __grid_constant__ CUtensorMap mB, GemmCrt g) {
    constexpr int kStages = Tile<kN>::kStages, kStageBytes = Tile<kN>::kStageBytes;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + kStages * kStageBytes);
    uint64_t *empty = full + kStages;
    uint64_t *cfull = empty + kStages;
    uint64_t *cfree = cfull + 2;
    uint64_t *done = cfree + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const uint32_t rank = cluster_rank();
    const bool lead = rank == 0;
    const int cl = static_cast<int>(blockIdx.x >> 1), ncl = static_cast<int>(gridDim.x >> 1);
    const int items = g.tiles * kMod * g.batch;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&cfull[b], 1);
            mbar_init(&cfree[b], 16);   // eight epilogue warps in each CTA of the pair
        }
        mbar_init(done, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(su32(tmem_slot)),
                     "r"(2 * kN));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;\n");
    }
    fence_before();
    __syncthreads();
    cluster_sync();
    fence_after();
    const uint32_t tmem = *tmem_slot;
    const int nk = (g.K + crt::kStageK - 1) / crt::kStageK;
    const int nchunks = (nk + crt::kChunk - 1) / crt::kChunk;

    // A wait of the whole warp, and whether it may go on: every lane gets the same answer.
    auto warp_wait = [&](uint64_t *bar, uint32_t parity) {
        const bool ok = __all_sync(0xffffffffu, mbar_wait_cl(bar, parity, g.err) && !*abort_flag);
        if (!ok) *abort_flag = 1;
        return ok;
    };
    if (warp == 8) {
        // ---- TMA: this CTA's rows of both operands, counted on the even CTA's full[s] ----
        const bool one = elected();
        bool ok = true;
        int issued = 0, kg = 0;
        const uint32_t full_pair = peer_addr(su32(&full[0]), 0);
        for (int w = cl; w < items && ok; w += ncl) {
            const int z = w / g.tiles;   // (batch item, modulus)
            int tm, tn;
            crt_tile(g, w - z * g.tiles, tm, tn);
            const int ya = tm * kTileM + static_cast<int>(rank) * 128, yb = tn * kN + static_cast<int>(rank) * (kN / 2);
            for (int kt = 0; kt < nk; ++kt, ++kg) {
                const int s = kg % kStages;
                if (kg >= kStages && !(ok = warp_wait(&empty[s], ((kg / kStages) & 1) ^ 1))) break;
                if (one) {
                    uint8_t *st = smem + s * kStageBytes;
                    if (lead) mbar_expect_tx(&full[s], 2 * kStageBytes);
                    const uint32_t fb = full_pair + static_cast<uint32_t>(s) * 8u;
                    tma_load_3d_pair(st, &mA, kt * crt::kStageK, ya, z, fb);
                    tma_load_3d_pair(st + kHalfBytes, &mB, kt * crt::kStageK, yb, z, fb);
                }
                __syncwarp();
                issued = kg + 1;
            }
        }
        if (!ok) {   // let the copies land before shared memory is released (as in k_tc.cu)
            if (lead) {
                for (int k = (issued > kStages ? issued - kStages : 0); k < issued; ++k)
                    mbar_wait_cl(&full[k % kStages], (k / kStages) & 1, g.err, kSpinCycles / 8);
            } else {
                const long long t0 = clock64();
                while (clock64() - t0 < 2000000LL) {
                }
            }
        }
    } else if (warp == 9) {
        if (lead) {
            const bool one = elected();
            bool ok = true;
            int kg = 0, cg = 0;
            for (int w = cl; w < items && ok; w += ncl, cg += nchunks) {
                for (int kt = 0; kt < nk; ++kt, ++kg) {
                    const int in = kt % crt::kChunk, c = cg + kt / crt::kChunk, buf = c & 1, s = kg % kStages;
                    if (in == 0 && c >= 2 && !(ok = warp_wait(&cfree[buf], ((c >> 1) - 1) & 1))) break;
                    if (!(ok = warp_wait(&full[s], (kg / kStages) & 1))) break;
                    fence_after();
                    const uint32_t base = su32(smem + s * kStageBytes), dt = tmem + static_cast<uint32_t>(buf * kN);
                    if (one) {
                        const uint64_t da = sdesc(base), db = sdesc(base + kHalfBytes);
#pragma unroll
                        for (int k = 0; k < 4; ++k)   // 32 bytes of K: two 16-byte units of the descriptor
                            mma_pair<kN>(dt, da + 2 * k, db + 2 * k, (in | k) != 0 ? 1u : 0u);
                        commit_both(su32(&empty[s]));
                        if (in == crt::kChunk - 1 || kt == nk - 1) commit_both(su32(&cfull[buf]));
                    }
                    __syncwarp();
                }
            }
            if (one) commit_both(su32(done));
            __syncwarp();
        }
    } else {
        // ---- epilogue: lane quarter q of this CTA's 128 rows, column half h; thread = row ----
        constexpr int kHalf = kN / 2;   // columns of a thread
        const int q = warp & 3, h = warp >> 2;
        const uint32_t cfree_pair = lead ? su32(&cfree[0]) : peer_addr(su32(&cfree[0]), 0);
        bool ok = true;
        int cg = 0;
        for (int w = cl; w < items && ok; w += ncl, cg += nchunks) {
            const int z = w / g.tiles;
            int tm, tn;
            crt_tile(g, w - z * g.tiles, tm, tn);
            const float m = c_m[z % kMod], back = c_back[z % kMod], inv = 1.0f / m;
            float acc[kHalf];
#pragma unroll
            for (int j = 0; j < kHalf; ++j) acc[j] = 0.f;
            for (int c = 0; c < nchunks; ++c) {
                const int buf = (cg + c) & 1;
                ok = mbar_wait_cl(&cfull[buf], ((cg + c) >> 1) & 1, g.err) && !*abort_flag;
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) {
                    *abort_flag = 1;
                    break;
                }
                fence_after();
                const uint32_t tb = tmem + (static_cast<uint32_t>(q * 32) << 16) + static_cast<uint32_t>(buf * kN + h * kHalf);
#pragma unroll
                for (int p = 0; p < kHalf / 32; ++p) {
                    uint32_t r[32];
                    tmem_ld32(tb + p * 32, r);
#pragma unroll
                    for (int j = 0; j < 32; ++j) acc[p * 32 + j] += crt::reduce(__uint_as_float(r[j]), m, inv);
                }
                fence_before();
                __syncwarp();
                if (lane == 0)
                    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];\n" ::"r"(
                                     cfree_pair + static_cast<uint32_t>(buf) * 8u)
                                 : "memory");
            }
            const long long row = static_cast<long long>(tm) * kTileM + rank * 128 + q * 32 + lane;
            if (!ok) break;
            uint8_t *y = g.Y + (static_cast<long long>(z) * g.M + row) * g.ldy;
            const int n0 = tn * kN + h * kHalf;
#pragma unroll
            for (int p = 0; p < kHalf / 16; ++p) {
                if (row >= g.M || n0 + 16 * p >= g.N) continue;   // ldy is a multiple of 16 not below N
                uint32_t v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    uint32_t b4[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        b4[j] = __float_as_uint(crt::stored(crt::reduce(acc[16 * p + 4 * u + j], m, inv), m, inv, back) + 8388608.0f);
                    v[u] = __byte_perm(__byte_perm(b4[0], b4[1], 0x0040), __byte_perm(b4[2], b4[3], 0x0040), 0x5410);
                }
                *reinterpret_cast<uint4 *>(y + n0 + 16 * p) = make_uint4(v[0], v[1], v[2], v[3]);
            }
            __syncwarp();   // the next tensor-memory load takes the whole warp
        }
    }
    __syncwarp();
    fence_before();
    __syncthreads();
    if (warp == 0) {
        if (lane == 0) mbar_wait_cl(done, 0, g.err);
        __syncwarp();
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(2 * kN));
    }
    __syncthreads();
    cluster_sync();
}

// ---- results --------------------------------------------------------------------------------
// A block of 256 threads takes kRows rows x 128 columns: a thread reads four neighbouring bytes of
// each of the 15 planes and sums them in three words (45 wide multiply-adds an entry, the FP64 pipe being
// the scarcer one: one conversion, three products).  Mirrored and transposed copies leave
// through shared memory, so that every store is a run of 256 bytes.
struct ResultArgs {
    const uint8_t *Y;
    long long ldy;
    const int *ea, *eb;      // [batch][a_rows], [batch][b_rows]
    int a_rows, b_rows, M, batch, n;      // n: columns of one part (all, or the complex product's half)
    int second;              // complex: first column of the imaginary part (0: real)
    double alpha, beta;
    const double *D;         // C and D: real plane, the imaginary one im_off further on
    double *C, *T;           // T: the transpose (null: none)
    long long ldd, ldc, ldt, sD, sC, sT, im_off;
    int col0;                // first column of C that this product covers
    int sym;                 // 0: all entries; 1: those on or above the diagonal, mirrored (the imaginary
                             // part with its sign changed); 2: those on or below it, not mirrored
};

__device__ __forceinline__ bool kept(int sym, int r, int c) { return sym == 0 || (sym == 1 ? c >= r : c <= r); }

template <int kRows>
__global__ void __launch_bounds__(256) k_crt_result(ResultArgs g, int tiles_c) {
    __shared__ double tile[kRows][129];
    const long long b = blockIdx.z;
    const int part = blockIdx.y;   // 0 real, 1 imaginary
    const int r0 = (blockIdx.x / tiles_c) * kRows, c0 = (blockIdx.x % tiles_c) * 128;
    if (g.sym == 1 ? g.col0 + c0 + 127 < r0 : g.sym && g.col0 + c0 > r0 + kRows - 1) return;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int c = c0 + 4 * tx, gc = g.col0 + c;
    double *C = g.C + b * g.sC + part * g.im_off;
    int eb[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) eb[j] = c + j < g.n ? g.eb[b * g.b_rows + part * g.second + c + j] : 0;
    const double unit = g.alpha * crt::kProduct;
    for (int i = ty; i < kRows; i += 8) {
        const int r = r0 + i;
        double v[4] = {0.0, 0.0, 0.0, 0.0};
        if (r < g.M && c < g.n) {
            const uint8_t *y = g.Y + (b * kMod * g.M + r) * g.ldy + part * g.second + c;
            crt::Words s[4];
            crt::each_modulus([&](auto I) {
                constexpr int k = decltype(I)::value;
                const uint32_t p = *reinterpret_cast<const uint32_t *>(y + k * g.M * g.ldy);
#pragma unroll
                for (int j = 0; j < 4; ++j) crt::accumulate<k>(s[j], (p >> (8 * j)) & 255u);
            });
            const int e = g.ea[b * g.a_rows + r];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                v[j] = crt::scaled_down(static_cast<double>(crt::fraction(s[j])) * unit, e, eb[j]);
                if (g.beta != 0.0 && c + j < g.n && kept(g.sym, r, gc + j))
                    v[j] += g.beta * g.D[b * g.sD + part * g.im_off + r * g.ldd + gc + j];
                if (g.sym && part && gc + j == r) v[j] = 0.0;   // a Hermitian result's diagonal is real
            }
            double *out = C + r * g.ldc + gc;
            if (c + 3 < g.n && kept(g.sym, r, gc) && kept(g.sym, r, gc + 3)) {
                reinterpret_cast<double2 *>(out)[0] = make_double2(v[0], v[1]);
                reinterpret_cast<double2 *>(out)[1] = make_double2(v[2], v[3]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (c + j < g.n && kept(g.sym, r, gc + j)) out[j] = v[j];
            }
        }
        if (g.sym == 1 || g.T) {
#pragma unroll
            for (int j = 0; j < 4; ++j) tile[i][4 * tx + j] = v[j];
        }
    }
    if (g.sym != 1 && !g.T) return;
    __syncthreads();
    const double sign = g.sym && part ? -1.0 : 1.0;
    double *out = g.sym ? C : g.T + b * g.sT + part * g.im_off;
    const long long ldo = g.sym ? g.ldc : g.ldt;
    constexpr int kGroups = 256 / kRows;   // columns of the tile at a time
    const int i = threadIdx.x % kRows, r = r0 + i;
    for (int k = threadIdx.x / kRows; k < 128; k += kGroups) {
        const int cc = g.col0 + c0 + k;
        if (r < g.M && c0 + k < g.n && (!g.sym || r < cc)) out[cc * ldo + r] = sign * tile[i][k];
    }
}

// Planes [z][rows][pitch] of bf16, boxes of box_rows rows by 64 entries of one plane, 128-byte swizzle.
bool plane_map(CUtensorMap *m, const void *base, long long K, long long rows, long long z, long long pitch,
               long long plane, int box_rows) {
    auto fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {static_cast<cuuint64_t>(K), static_cast<cuuint64_t>(rows), static_cast<cuuint64_t>(z)};
    cuuint64_t strides[2] = {static_cast<cuuint64_t>(2 * pitch), static_cast<cuuint64_t>(2 * plane)};
    cuuint32_t box[3] = {crt::kStageK, static_cast<cuuint32_t>(box_rows), 1};
    cuuint32_t es[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

inline long long up(long long x, long long m) { return (x + m - 1) / m * m; }

}  // namespace

// ---- host -----------------------------------------------------------------------------------
CrtShape crt_shape(int rows, int K, int batch, bool complex, bool right) {
    CrtShape s;
    s.rows = rows;
    s.K = K;
    s.batch = batch;
    s.half = static_cast<int>(up(K, 64));   // rows on 128-byte lines
    s.second = complex && right ? static_cast<int>(up(rows, 16)) : 0;
    s.out_rows = rows + s.second;
    s.pitch = complex ? 2LL * s.half : s.half;
    s.complex = complex;
    s.right = right;
    return s;
}

size_t crt_operand_bytes(const CrtShape &s) {
    return static_cast<size_t>(up(2LL * kMod * s.batch * s.out_rows * s.pitch, 256) + up(4LL * s.batch * s.out_rows, 256));
}
size_t crt_bytes_bytes(int M, int N, int batch) { return static_cast<size_t>(up(kMod * static_cast<long long>(batch) * M * up(N, 16), 256)); }

CrtOperand crt_rows(const CrtShape &s, const double *re, const double *im, long long ld, long long stride, bool conj,
                    void *mem, cudaStream_t st) {
    const long long plane = s.out_rows * s.pitch;
    CrtOperand o{s, plane, s.out_rows, static_cast<__nv_bfloat16 *>(mem),
                 reinterpret_cast<int *>(static_cast<char *>(mem) + up(2LL * kMod * s.batch * plane, 256))};
    RowsArgs g{re, s.complex ? im : nullptr, ld, stride, s.rows, s.K, s.right, conj, s.half, s.second, o.planes, s.pitch,
               plane, kMod * plane, o.exps, s.out_rows};
    count_launches(1);
    // a warp per row up to 512 entries; longer rows would leave a warp too long alone with one
    if (s.K <= 512) k_crt_rows<32><<<dim3((s.rows + 3) / 4, s.batch), 128, 0, st>>>(g);
    else k_crt_rows<128><<<dim3(s.rows, s.batch), 128, 0, st>>>(g);
    return o;
}

namespace {

template <int kN>
cudaError_t launch_gemm(const CrtOperand &A, const CrtOperand &B, GemmCrt &g, cudaStream_t st) {
    const CrtShape &a = A.shape, &b = B.shape;
    CUtensorMap ma, mb;
    const long long z = static_cast<long long>(kMod) * a.batch;
    if (!plane_map(&ma, A.planes, g.K, a.out_rows, z, a.pitch, A.plane, 128) ||
        !plane_map(&mb, B.planes, g.K, b.out_rows, z, b.pitch, B.plane, kN / 2))
        return cudaErrorInvalidValue;
    g.tiles_m = (g.M + kTileM - 1) / kTileM;
    g.tiles_n = (g.N + kN - 1) / kN;
    g.tiles = g.half ? g.tiles_n * (g.tiles_n + 1) / 2 : g.tiles_m * g.tiles_n;
    static std::atomic<int> resident{0};   // clusters at one time, the same for every device of this kind
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.blockDim = dim3(32 * kWarps);
    cfg.dynamicSmemBytes = Tile<kN>::kSmem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaFuncSetAttribute(k_crt_gemm<kN>, cudaFuncAttributeMaxDynamicSharedMemorySize, Tile<kN>::kSmem);
    if (e != cudaSuccess) return e;
    int most = resident.load();
    if (!most) {
        int dev = 0, sms = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cfg.gridDim = dim3(static_cast<unsigned>(sms & ~1));
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&most, k_crt_gemm<kN>, &cfg);
        if (e != cudaSuccess) return e;
        if (most < 1) return cudaErrorInvalidConfiguration;
        resident.store(most);
    }
    const long long items = static_cast<long long>(g.tiles) * kMod * a.batch;
    cfg.gridDim = dim3(static_cast<unsigned>(2 * std::min<long long>(items, most)));
    count_launches(1);
    return cudaLaunchKernelEx(&cfg, k_crt_gemm<kN>, ma, mb, g);
}

}  // namespace

cudaError_t crt_products(const CrtOperand &A, const CrtOperand &B, int M, int half, void *bytes, int *err,
                         cudaStream_t st) {
    GemmCrt g{};
    g.M = M;
    g.N = B.shape.out_rows;
    g.K = static_cast<int>(A.shape.K);
    if (A.shape.complex) g.K = static_cast<int>(A.shape.pitch);
    g.batch = A.shape.batch;
    g.half = half;
    g.Y = static_cast<uint8_t *>(bytes);
    g.ldy = up(g.N, 16);
    g.err = err;
    // narrow tiles where wide ones would be mostly padding, or too few to go round
    if (g.N <= 128) {
        g.half = 0;
        return launch_gemm<64>(A, B, g, st);
    }
    return launch_gemm<256>(A, B, g, st);
}

cudaError_t crt_multiply(const CrtOperand &A, const CrtOperand &B, const CrtResult &r, void *bytes, int *err,
                         cudaStream_t st) {
    const CrtShape &a = A.shape, &b = B.shape;
    if (a.K != b.K || a.batch != b.batch || a.complex != b.complex || (a.complex && (a.right || !b.right)))
        return cudaErrorInvalidValue;
    // a symmetric result's upper half needs the rows above its last column only
    const int M = r.sym == 1 ? std::min(a.rows, r.col0 + b.rows) : a.rows, N = b.out_rows;
    const bool square = !a.complex && M == N && r.col0 == 0;
    const cudaError_t e = crt_products(A, B, M, square ? r.sym : 0, bytes, err, st);
    if (e != cudaSuccess) return e;
    ResultArgs o{};
    o.Y = static_cast<const uint8_t *>(bytes);
    o.ldy = up(N, 16);
    o.ea = A.exps;
    o.eb = B.exps;
    o.a_rows = A.exp_stride;
    o.b_rows = B.exp_stride;
    o.M = M;
    o.batch = a.batch;
    o.n = b.rows;
    o.second = b.second;
    o.alpha = r.alpha;
    o.beta = r.beta;
    o.D = r.D;
    o.C = r.C;
    o.T = r.T;
    o.ldd = r.ldd;
    o.ldc = r.ldc;
    o.ldt = r.ldt;
    o.sD = r.sD;
    o.sC = r.sC;
    o.sT = r.sT;
    o.im_off = r.im_off;
    o.col0 = r.col0;
    o.sym = r.sym;
    const int tc = (o.n + 127) / 128, z = (a.complex ? 2 : 1) * a.batch;
    const dim3 rest(1, a.complex ? 2 : 1, a.batch);
    count_launches(1);
    // blocks of 8 rows, one a warp, until they fill the chip twice (order 96: 15.6 us with 32 rows, 6.1 with 8)
    if ((M + 31) / 32 * tc * z >= 2 * 152) {
        k_crt_result<32><<<dim3((M + 31) / 32 * tc, rest.y, rest.z), 256, 0, st>>>(o, tc);
    } else {
        k_crt_result<8><<<dim3((M + 7) / 8 * tc, rest.y, rest.z), 256, 0, st>>>(o, tc);
    }
    return cudaGetLastError();
}

size_t crt_gemm_bytes(int M, int N, int K, int panel) {
    const int kb = std::min(K, panel), nb = std::min(N, panel);
    return crt_operand_bytes(crt_shape(M, kb, 1, false, false)) + crt_operand_bytes(crt_shape(nb, kb, 1, false, true)) +
           crt_bytes_bytes(M, nb, 1);
}

cudaError_t crt_gemm(const double *A, long long lda, const double *Bt, long long ldb, int M, int N, int K,
                     const CrtResult &r, void *work, int *err, cudaStream_t st, int panel) {
    for (int k0 = 0; k0 < K; k0 += panel) {
        const int kb = std::min(K - k0, panel);
        char *p = static_cast<char *>(work);
        const CrtShape sa = crt_shape(M, kb, 1, false, false);
        const CrtOperand a = crt_rows(sa, A + k0, nullptr, lda, 0, false, p, st);
        p += crt_operand_bytes(sa);
        for (int n0 = 0; n0 < N; n0 += panel) {
            const int nb = std::min(N - n0, panel);
            const CrtShape sb = crt_shape(nb, kb, 1, false, true);
            const CrtOperand b = crt_rows(sb, Bt + n0 * ldb + k0, nullptr, ldb, 0, false, p, st);
            CrtResult rp = r;
            rp.col0 = n0;
            if (k0) {
                rp.beta = 1.0;
                rp.D = r.C;
                rp.ldd = r.ldc;
            }
            if (k0 + kb < K) rp.T = nullptr;
            const cudaError_t e = crt_multiply(a, b, rp, p + crt_operand_bytes(sb), err, st);
            if (e != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

}  // namespace mbdgb
