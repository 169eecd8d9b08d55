// Host orchestration and C ABI of libmbdgb (declared in include/mbd_gb300.h).
//
// One evaluation is one stream-ordered pass over the device:
//   prepare_atoms -> build_scs (all frequencies) -> batched Cholesky -> X = A^{-1} E
//   -> contract_screen -> build_q -> Gershgorin scale -> coupled Newton-Schulz
//   -> energy; and for gradients: mbd_grad_pass -> chain_screen -> V = A^{-1} H
//   -> scs_grad_pass -> ts_chain.
// The host reads back one scalar per Newton-Schulz iteration (the convergence test)
// and the status word after the screening stage.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/mbd_gb300.h"
#include "../../include/mbd_gb300_kernels.h"
#include <nvtx3/nvToolsExt.h>

#include "internal.h"
#include "freq_grid.h"
#include "ns_schedule.h"

using namespace mbdgb;

namespace {
std::atomic<long long> g_launches{0};
// Refinement steps of the mixed screening solves: the FP32 factor's solution carries relative
// errors of a few 1e-7 in the screened polarizabilities, one step against the FP64 matrix
// brings them to about 1e-13 (screening matrices of kappa up to ~2e3).
constexpr int kRefineSteps = 1;
// Refinement steps of the mixed modes' adjoint solves V = A^{-1} H: the unrefined FP32 solve
// errs by at most kappa(A) eps32 ~ 1e-4 relative to the SCS part of the gradient; the TF32x3
// force error measured at 2000 atoms with it (3e-6 of the largest force) is well inside that.
constexpr int kAdjointRefineSteps = 0;
constexpr int kLanczosSteps = 48; // Lanczos steps of the spectrum estimate of Q
// ... and in the mixed modes for Q of order <= kLanczosSmallOrder: on the spectra of clusters of
// 70-500 atoms the mixed loop, which stops at its precision floor, takes the same number of
// steps (8-9) from a 24-step estimate as from a 48-step one (the lower estimate is then 3-10
// times higher, which only shortens the first steps), while the 24 steps save 48 of the
// evaluation's ~190 launches.  The FP64 loop, which converges further, can take one step
// more from it (11 against 10 on a 500-atom cluster) and keeps the 48.
constexpr int kLanczosStepsSmall = 24;
constexpr long long kLanczosSmallOrder = 2048;
// Precision floor of the TF32x3 Newton-Schulz iteration per unit of sqrt(n): |I - Z Y|_F
// settles at about 1.04e-7 sqrt(n) (8.1e-6 at n = 6000).  A step taken from a residual r whose
// exact successor bound 0.875 r^2 lies below this is the last useful one.  The coarser kinds
// (TF32, BF16x3) reach their floors above it and stop by the halving test alone.
constexpr double kMixedFloor = 1e-7;
// Periodic Newton-Schulz (FP64): Y' and Z' as Hermitian products (upper tiles only, real part
// mirrored, imaginary part mirrored with a sign change), a third fewer flops per step.
constexpr bool kHermitianNs = true;
constexpr int kLF = MBD_LEARNED_FEATURES;   // inputs of the learned screening model
// The FP64 path (screening, bounds, Newton-Schulz, gradients in FP64).
inline bool fp64_path(int precision) { return precision == MBD_PREC_FP64 || precision == MBD_PREC_FP64_SPLIT; }
}  // namespace

void mbdgb::count_launches(int k) { g_launches.fetch_add(k, std::memory_order_relaxed); }
long long mbdgb::launch_count() { return g_launches.load(std::memory_order_relaxed); }

namespace {

// Number of eigenvalues below x of the symmetric tridiagonal matrix (diag a, offdiag b)
// by the Sturm sequence of its LDL^T pivots.
int sturm_count(const std::vector<double> &a, const std::vector<double> &b, double x) {
    int cnt = 0;
    double d = 1.0;
    for (size_t i = 0; i < a.size(); ++i) {
        const double off = i ? b[i - 1] * b[i - 1] : 0.0;
        d = a[i] - x - (i ? off / d : 0.0);
        if (d == 0.0) d = -1e-300;
        if (d < 0.0) ++cnt;
    }
    return cnt;
}

// Smallest and largest eigenvalue of a symmetric tridiagonal matrix by bisection.
void tridiag_extremes(const std::vector<double> &a, const std::vector<double> &b, double &lo, double &hi) {
    double g0 = 1e300, g1 = -1e300;   // Gershgorin interval of the tridiagonal
    for (size_t i = 0; i < a.size(); ++i) {
        const double r = (i ? std::fabs(b[i - 1]) : 0.0) + (i + 1 < a.size() ? std::fabs(b[i]) : 0.0);
        g0 = std::min(g0, a[i] - r);
        g1 = std::max(g1, a[i] + r);
    }
    const int m = static_cast<int>(a.size());
    double l = g0, h = g1;
    for (int it = 0; it < 200; ++it) {   // smallest: count(x) >= 1
        const double mid = 0.5 * (l + h);
        if (mid == l || mid == h) break;   // the interval is one rounding wide
        if (sturm_count(a, b, mid) >= 1) h = mid; else l = mid;
    }
    lo = h;
    l = g0; h = g1;
    for (int it = 0; it < 200; ++it) {   // largest: count(x) >= m
        const double mid = 0.5 * (l + h);
        if (mid == l || mid == h) break;
        if (sturm_count(a, b, mid) >= m) h = mid; else l = mid;
    }
    hi = h;
}

}  // namespace

struct mbd_ctx {
    int device = 0;
    mbd_options opt{};
    cudaStream_t stream = nullptr;
    // problem
    int N = 0, n = 0, nf1 = 0, nb = 0;
    long long ld = 0;
    bool have_geom = false, have_params = false;
    std::vector<double> hR, ha0, hc6, hrr, hv;
    std::vector<double> hu, hwu;
    // device memory: one slab, carved
    void *slab = nullptr;
    size_t slab_bytes = 0;
    ScratchLimits lim;
    double *dR, *da0ref, *dc6ref, *drref, *dratio;
    double *da0, *dom, *drv, *dalu, *dsigu, *dabar, *dabar0, *dc6bar, *dombar, *drbar, *du, *dwu;
    double *dM, *ddinv, *dX, *dV, *dB;
    float *sM = nullptr, *sdinv = nullptr, *swork = nullptr;   // FP32 factors of the mixed modes
    uint32_t *spanel = nullptr;   // TF32x3 parts of the factor panels (tensor-core trailing updates)
    float *sgrad32 = nullptr;     // FP32 inputs of the reduced-precision SCS adjoint pair pass
    double *dlog = nullptr;       // per-frequency sums of the log-formula route: ln det, Tr A^2..4
    double *dtq = nullptr;        // Tr (Q^{1/2})_ii per atom from the mixed modes' FP64 correction
    bool tq_valid = false;
    double *dQ, *dZ, *dP, *dY2, *dZ2;
    // mixed-precision Newton-Schulz buffers (ld x ld each)
    float *fY = nullptr, *fZ = nullptr, *fY2 = nullptr, *fZ2 = nullptr, *fP = nullptr, *fPT = nullptr;
    void *hY[2] = {}, *hZ[2] = {}, *hY2[2] = {}, *hZ2[2] = {}, *hP[2] = {}, *hPT[2] = {};   // split operands
    double corr_resid = 0.0;   // |Zd Q Zd - I|_F of the mixed modes' correction
    // mixed modes on a cell: each Hermitian Q(q) as the real symmetric [[Re, -Im], [Im, Re]] of
    // order 2n (leading dimension lde), its FP64 workspaces
    long long lde = 0;
    int mgroup = 1;   // Bloch vectors iterated on together, of which the FP32, split and e* buffers hold one matrix each
    double *dmix = nullptr;   // per matrix of a group: |I - ZY|^2, the correction's residual, the largest row sum
    double *eM = nullptr, *eV = nullptr, *eW = nullptr, *eVT = nullptr, *eZ = nullptr;
    double *dh, *dgomb, *dgab0, *dgrb, *dgR, *dga0, *dgom, *dgrv, *dgp;
    // periodic systems: cell, Bloch vectors and reciprocal lattice (host lists, device copies)
    bool periodic = false;
    int nk = 1, nG = 0, maxG = 0;
    int nkt = 1;   // Bloch vectors of the whole grid, of which nk are kept (with weights hkw, the sum nkt)
    CellGeom cell{};
    std::vector<double> hkq, hkw, hG;
    std::vector<int> hglist, hgcount;
    // FP64 path: residue planes of three operands and the bytes of a product (k_crt.cu), or the
    // scratch of products taken in panels; dPT: the transpose of P.  Null when they did not fit:
    // the products then run on the FP64 pipe.
    char *crt = nullptr;
    double *dPT = nullptr;
    char *qwork = nullptr;   // cells: scratch of the Q(q) build's products (null: it runs on the FP64 pipe)
    size_t qwork_bytes = 0;
    void *qslab = nullptr;   // qwork's own memory, once a changed lattice needed more than the slab's
    bool no_scratch = false;   // the scratch of the tensor-core products did not fit the card
    double *dkq = nullptr, *dkw = nullptr, *dG = nullptr, *dcoef = nullptr, *dlzw = nullptr, *dgA = nullptr, *dgAout = nullptr,
           *dgApart = nullptr, *dgc = nullptr, *dtsg = nullptr;
    int *dglist = nullptr, *dgcount = nullptr;
    double2 *dS = nullptr;
    bool have_lattice_grad = false;
    // learned screening model (host copy; device buffers in their own allocation)
    int members = 0;
    std::vector<uint16_t> hmodel;
    std::vector<float> hmean, hstd;
    bool model_dirty = false, force_plain = false;
    void *lslab = nullptr;
    size_t lbytes = 0;
    int lN = 0, lM = 0;
    void *dmodel = nullptr;
    float *dmeanstd = nullptr, *dfeat = nullptr, *dYl = nullptr;
    double *dspread = nullptr, *dmoments = nullptr, *dadj = nullptr;
    float *dzc = nullptr, *dXl = nullptr;   // MLP cache and feature gradient (learned forces)
    float *dpacked = nullptr;               // the members' weights in the MLP kernels' layout
    int *doffs = nullptr;
    double learned_est = 0.0;
    int learned_fallback = 0;
    bool last_learned = false;   // the last forward kept the learned model's screening
    double *dscal;   // [0] energy, [1] Gershgorin, [2] residual
    int *dstatus;
    // last results
    int ns_iter = 0;
    double ns_scale = 0.0, ns_resid = 0.0;
    bool have_result = false;
    bool have_screening = false;
    // state of the last forward evaluation, kept for mbd_backward_dev
    bool have_forward = false;
    long long eval_count = 0;  // successful evaluations of this context so far
    double *Zlast = nullptr;   // Newton-Schulz Z (Q^{-1/2} = zscale * Z)
    double zscale = 0.0;
    // exception
    int err_code = MBD_OK;
    std::string err_origin, err_msg;
    // profiling (CUDA events on the launch stream)
    bool profiling = false;
    std::vector<cudaEvent_t> events;
    int ev_used = 0;
    mbd_profile prof{};
};

namespace {

int fail(mbd_ctx *c, int code, const char *origin, const std::string &msg) {
    if (c) {
        c->err_code = code;
        c->err_origin = origin;
        c->err_msg = msg;
    }
    return code;
}

int cuda_fail(mbd_ctx *c, const char *origin, cudaError_t e) {
    return fail(c, MBD_ERR_CUDA, origin, std::string("CUDA error: ") + cudaGetErrorString(e));
}

#define MBD_CUDA(call, origin)                                  \
    do {                                                        \
        cudaError_t e_ = (call);                                \
        if (e_ != cudaSuccess) return cuda_fail(ctx, origin, e_); \
    } while (0)

// Next free timing event of the context (created on first use, reused per evaluation).
cudaEvent_t next_event(mbd_ctx *ctx) {
    if (ctx->ev_used == static_cast<int>(ctx->events.size())) {
        cudaEvent_t e;
        if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
        ctx->events.push_back(e);
    }
    return ctx->events[ctx->ev_used++];
}

struct Span { cudaEvent_t a = nullptr, b = nullptr; double flops = 0.0; };

// NVTX ranges of the evaluation stages on the host timeline (no-ops unless a profiler is
// attached); the range open at any return is closed by the destructor.
struct NvtxStages {
    bool open = false;
    void next(const char *name) {
        if (open) nvtxRangePop();
        nvtxRangePushA(name);
        open = true;
    }
    ~NvtxStages() {
        if (open) nvtxRangePop();
    }
};

void mark(mbd_ctx *ctx, cudaStream_t s, cudaEvent_t &e) {
    if (!ctx->profiling) return;
    e = next_event(ctx);
    if (e) cudaEventRecord(e, s);
}

double span_ms(cudaEvent_t a, cudaEvent_t b) {
    float ms = 0.f;
    if (a && b && cudaEventElapsedTime(&ms, a, b) == cudaSuccess) return ms;
    return 0.0;
}

void release(mbd_ctx *ctx) {
    if (ctx->slab) cudaFree(ctx->slab);
    ctx->slab = nullptr;
    if (ctx->qslab) cudaFree(ctx->qslab);
    ctx->qslab = nullptr;
    ctx->slab_bytes = 0;
}

// Device buffers of the learned model for N atoms and M members (own allocation, resized on
// demand); uploads the model when it changed.
int ensure_learned(mbd_ctx *ctx) {
    const int N = ctx->N, M = ctx->members, nf1 = ctx->nf1;
    const size_t P = static_cast<size_t>(learned_param_count());
    auto al = [](size_t b) { return (b + 255) / 256 * 256; };
    if (!ctx->lslab || ctx->lN != N || ctx->lM != M) {
        const size_t bytes = al(2 * P * M) + al(sizeof(float) * 2 * kLF) + al(sizeof(float) * kLF * N) +
                             al(sizeof(float) * M * N * 16) + al(sizeof(double) * nf1 * N) +
                             al(sizeof(double) * kLearnedWork * N) + al(sizeof(double) * kLearnedAdjointWork * N) +
                             al(sizeof(float) * M * 2 * N * 128) +
                             al(sizeof(float) * M * N * kLF) + al(sizeof(float) * M * kLearnedPackedFloats) +
                             al(sizeof(int) * 2);
        cudaError_t e = cudaSuccess;
        if (!ctx->lslab || ctx->lbytes < bytes) {   // re-carved in place when large enough
            if (ctx->lslab) cudaFree(ctx->lslab);
            ctx->lslab = nullptr;
            e = cudaMalloc(&ctx->lslab, bytes);
            if (e != cudaSuccess) return cuda_fail(ctx, "learned_screening", e);
            ctx->lbytes = bytes;
        }
        char *p = static_cast<char *>(ctx->lslab);
        ctx->dmodel = p; p += al(2 * P * M);
        ctx->dmeanstd = reinterpret_cast<float *>(p); p += al(sizeof(float) * 2 * kLF);
        ctx->dfeat = reinterpret_cast<float *>(p); p += al(sizeof(float) * kLF * N);
        ctx->dYl = reinterpret_cast<float *>(p); p += al(sizeof(float) * M * N * 16);
        ctx->dspread = reinterpret_cast<double *>(p); p += al(sizeof(double) * nf1 * N);
        ctx->dmoments = reinterpret_cast<double *>(p); p += al(sizeof(double) * kLearnedWork * N);
        ctx->dadj = reinterpret_cast<double *>(p); p += al(sizeof(double) * kLearnedAdjointWork * N);
        ctx->dzc = reinterpret_cast<float *>(p); p += al(sizeof(float) * M * 2 * N * 128);
        ctx->dXl = reinterpret_cast<float *>(p); p += al(sizeof(float) * M * N * kLF);
        ctx->dpacked = reinterpret_cast<float *>(p); p += al(sizeof(float) * M * kLearnedPackedFloats);
        ctx->doffs = reinterpret_cast<int *>(p);
        const int offs[2] = {0, N};
        e = cudaMemcpy(ctx->doffs, offs, sizeof(offs), cudaMemcpyHostToDevice);
        if (e != cudaSuccess) return cuda_fail(ctx, "learned_screening", e);
        ctx->lN = N;
        ctx->lM = M;
        ctx->model_dirty = true;
    }
    if (ctx->model_dirty) {
        cudaError_t e = cudaMemcpy(ctx->dmodel, ctx->hmodel.data(), 2 * P * M, cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemcpy(ctx->dmeanstd, ctx->hmean.data(), sizeof(float) * kLF, cudaMemcpyHostToDevice);
        if (e == cudaSuccess)
            e = cudaMemcpy(ctx->dmeanstd + kLF, ctx->hstd.data(), sizeof(float) * kLF, cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = mlp_pack(M, ctx->dmodel, ctx->dpacked, nullptr);
        if (e == cudaSuccess) e = cudaDeviceSynchronize();
        if (e != cudaSuccess) return cuda_fail(ctx, "learned_screening", e);
        ctx->model_dirty = false;
    }
    return MBD_OK;
}

// Scratch of the FP64 path's products for matrices of order n: three operands' residue planes and a
// product's bytes while a matrix is one panel, else that of products in panels.
size_t crt_ns_bytes(int n, const ScratchLimits &lim) {
    if (n > lim.panel) return crt_gemm_bytes(n, n, n, lim.panel);
    return 3 * crt_operand_bytes(crt_shape(n, n, 1, false, false)) + crt_bytes_bytes(n, n, 1);
}

// The products of a coupled Newton-Schulz step on the tensor cores (k_crt.cu).  All operands are
// rows: Y and Z are symmetric, and P's columns are the rows of its transpose, which P's own
// product writes beside it.  Each matrix becomes residue planes once a step.
struct CrtProducts {
    mbd_ctx *ctx;
    cudaStream_t s;
    CrtShape shape;
    char *slot[3], *bytes;
    CrtOperand oY{}, oZ{};
    CrtProducts(mbd_ctx *c, cudaStream_t st) : ctx(c), s(st), shape(crt_shape(c->n, c->n, 1, false, false)) {
        const size_t b = crt_operand_bytes(shape);
        for (int k = 0; k < 3; ++k) slot[k] = c->crt + k * b;
        bytes = c->crt + 3 * b;
    }
    bool panels() const { return ctx->n > ctx->lim.panel; }
    CrtOperand rows(const double *X, int k) { return crt_rows(shape, X, nullptr, ctx->ld, 0, false, slot[k], s); }
    CrtResult result(double *C, double *T, double alpha, double beta, const double *D, bool sym) const {
        const long long ld = ctx->ld;
        return CrtResult{alpha, beta, D, C, T, ld, ld, ld, 0, 0, 0, 0, 0, sym ? 1 : 0};
    }
    cudaError_t whole(const double *A, const double *Bt, const CrtResult &r) {
        return crt_gemm(A, ctx->ld, Bt, ctx->ld, ctx->n, ctx->n, ctx->n, r, ctx->crt, ctx->dstatus, s, ctx->lim.panel);
    }
    // P = Z Y and its transpose
    cudaError_t product(const double *Z, const double *Y, double *P, double *PT) {
        const CrtResult r = result(P, PT, 1.0, 0.0, nullptr, false);
        if (panels()) return whole(Z, Y, r);
        oZ = rows(Z, 0);
        oY = rows(Y, 1);
        return crt_multiply(oZ, oY, r, bytes, ctx->dstatus, s);
    }
    // Y2 = c1 Y + c3 Y P, Z2 = c1 Z + c3 P Z, after product()
    cudaError_t step(const double *Y, const double *Z, const double *P, const double *PT, double *Y2, double *Z2,
                     double c1, double c3) {
        const CrtResult ry = result(Y2, nullptr, c3, c1, Y, true), rz = result(Z2, nullptr, c3, c1, Z, true);
        if (panels()) {
            const cudaError_t e = whole(Y, PT, ry);
            return e == cudaSuccess ? whole(P, Z, rz) : e;
        }
        const cudaError_t e = crt_multiply(oY, rows(PT, 2), ry, bytes, ctx->dstatus, s);
        return e == cudaSuccess ? crt_multiply(rows(P, 1), oZ, rz, bytes, ctx->dstatus, s) : e;
    }
    // Y2 = c1 Y + c3 Y Y
    cudaError_t first_step(const double *Y, double *Y2, double c1, double c3) {
        const CrtResult r = result(Y2, nullptr, c3, c1, Y, true);
        if (panels()) return whole(Y, Y, r);
        oY = rows(Y, 1);
        return crt_multiply(oY, oY, r, bytes, ctx->dstatus, s);
    }
};

// Bloch vectors per complex product, and its scratch.
int crt_cell_group(int n, int nk, const ScratchLimits &lim) {
    const size_t one = crt_operand_bytes(crt_shape(n, n, 1, true, false)) +
                       crt_operand_bytes(crt_shape(n, n, 1, true, true)) +
                       crt_bytes_bytes(n, crt_shape(n, n, 1, true, true).out_rows, 1);
    return static_cast<int>(std::min<size_t>(nk, std::max<size_t>(1, lim.cell_products / one)));
}
size_t crt_cell_bytes(int n, int nk, const ScratchLimits &lim) {
    const int g = crt_cell_group(n, nk, lim);
    return crt_operand_bytes(crt_shape(n, n, g, true, false)) + crt_operand_bytes(crt_shape(n, n, g, true, true)) +
           crt_bytes_bytes(n, crt_shape(n, n, g, true, true).out_rows, g);
}

// C = alpha A B + beta D for the planar complex matrices of every Bloch vector, B from the rows of B^T
// (conj: from the rows of a Hermitian B); T: also the transpose; sym: Hermitian results.
cudaError_t crt_cell_product(mbd_ctx *ctx, const double *A, const double *Bt, bool conj, const double *D, double *C,
                             double *T, double alpha, double beta, bool sym, cudaStream_t s) {
    const int n = ctx->n, group = crt_cell_group(n, ctx->nk, ctx->lim);
    const long long ld = ctx->ld, m2 = ld * ld, st = 2 * m2;
    for (int k0 = 0; k0 < ctx->nk; k0 += group) {
        const int g = std::min(group, ctx->nk - k0);
        const CrtShape sa = crt_shape(n, n, g, true, false), sb = crt_shape(n, n, g, true, true);
        char *pb = ctx->crt + crt_operand_bytes(sa);
        const CrtOperand a = crt_rows(sa, A + k0 * st, A + k0 * st + m2, ld, st, false, ctx->crt, s);
        const CrtOperand b = crt_rows(sb, Bt + k0 * st, Bt + k0 * st + m2, ld, st, conj, pb, s);
        const CrtResult r{alpha, beta, D ? D + k0 * st : nullptr, C + k0 * st, T ? T + k0 * st : nullptr,
                          ld, ld, ld, st, st, st, m2, 0, sym ? 1 : 0};
        const cudaError_t e = crt_multiply(a, b, r, pb + crt_operand_bytes(sb), ctx->dstatus, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// FP64 factors of a batch of matrices: on the tensor cores where their scratch is there.
int factorise(mbd_ctx *ctx, double *A, int batch, cudaStream_t s, const char *origin) {
    const long long ld = ctx->ld;
    if (!ctx->crt) {
        cholesky_f64(A, ld, ld * ld, batch, ctx->ddinv, ctx->dstatus, s);
        return MBD_OK;
    }
    MBD_CUDA(cholesky_crt(A, ld, ld * ld, batch, ctx->ddinv, ctx->crt, ctx->dstatus, s, ctx->lim), origin);
    return MBD_OK;
}

// Bloch vectors that the mixed modes iterate on together: enough for eight tiles of a symmetric product
// on every SM, while their matrices take at most 4 GiB.  Alone, a matrix of the 256-atom cell (order 1536: 42
// tiles) leaves most of the 152 SMs idle, and each of its launches and read-backs serves one matrix.
int mixed_group(int nk, long long lde, int precision) {
    const long long t = lde / 128, tiles = (t + 1) * (t + 1) / 4;   // 128 x 256 tiles of one triangle
    const long long split = precision == MBD_PREC_BF16X3 ? 24 : (precision == MBD_PREC_TF32X3 ? 48 : 0);
    const long long bytes = lde * lde * (6 * 4 + 5 * 8 + split);
    const long long want = std::min<long long>((8 * 152 + tiles - 1) / tiles, (4LL << 30) / bytes);
    return static_cast<int>(std::max<long long>(1, std::min<long long>({want, nk, kTcSlots})));
}

// Scratch of a cell's products: the gradient's and, in FP64, those that build Q(q).  (The mixed modes round Q to FP32 and
// bf16 parts, where a last-place difference of the FP64 entries now and then turns a rounding, and keep the direct build:
// through products their 256-atom cell takes 150 ms less, but one in five seeds comes out 5e-9 off.)
size_t cell_products_bytes(int N, const CellGeom &c, int nk, int maxG, int precision, const ScratchLimits &lim) {
    const size_t grad = grad_products_bytes(N, c, nk, maxG, lim);
    return fp64_path(precision) ? std::max(build_q_products_bytes(N, c, nk, maxG, lim), grad) : grad;
}

// Carves the workspace out of one allocation (256-byte aligned pieces).
int allocate(mbd_ctx *ctx, bool groups = true) {
    const long long ld = ctx->ld, N = ctx->N, nf1 = ctx->nf1, nb = ctx->nb;
    const size_t mat = sizeof(double) * static_cast<size_t>(ld) * ld;
    std::vector<std::pair<double **, size_t>> plan = {
        {&ctx->dR, 3 * N}, {&ctx->da0ref, N}, {&ctx->dc6ref, N}, {&ctx->drref, N}, {&ctx->dratio, N},
        {&ctx->da0, N}, {&ctx->dom, N}, {&ctx->drv, N}, {&ctx->dalu, nf1 * N}, {&ctx->dsigu, nf1 * N},
        {&ctx->dabar, nf1 * N}, {&ctx->dabar0, N}, {&ctx->dc6bar, N}, {&ctx->dombar, N},
        {&ctx->drbar, N}, {&ctx->du, nf1}, {&ctx->dwu, nf1}, {&ctx->dlog, 4 * nf1}, {&ctx->dtq, N},
        {&ctx->ddinv, nf1 * nb * 4096}, {&ctx->dX, nf1 * ld * 3}, {&ctx->dV, nf1 * ld * 3},
        {&ctx->dB, nf1 * ld * 3},
        {&ctx->dh, nf1 * N}, {&ctx->dgomb, N}, {&ctx->dgab0, N}, {&ctx->dgrb, N}, {&ctx->dgR, 3 * N},
        {&ctx->dga0, N}, {&ctx->dgom, N}, {&ctx->dgrv, N}, {&ctx->dgp, 4 * N}, {&ctx->dscal, 8 + 2 * 64 + 1824},
        {&ctx->dmix, 3 * kTcSlots},
    };
    const long long nk = ctx->nk;
    if (ctx->periodic) {
        plan.push_back({&ctx->dkq, 3 * nk});
        plan.push_back({&ctx->dkw, nk});
        plan.push_back({&ctx->dG, 3LL * ctx->nG});
        plan.push_back({&ctx->dcoef, nk * (2 * kLanczosSteps + 1)});   // and the mixed modes' energies
        plan.push_back({&ctx->dlzw, 3 * nk * 2 * ld});
        plan.push_back({&ctx->dgA, 9});
        plan.push_back({&ctx->dgAout, 9});
        plan.push_back({&ctx->dgApart, scs_grad_periodic_words(static_cast<int>(N), static_cast<int>(nf1))});
        plan.push_back({&ctx->dgc, N});
        plan.push_back({&ctx->dtsg, 2LL * ctx->nG});
        plan.push_back({reinterpret_cast<double **>(&ctx->dS), 2LL * ctx->nG * N});
        plan.push_back({reinterpret_cast<double **>(&ctx->dglist), (nk * ctx->maxG + 1) / 2});
        plan.push_back({reinterpret_cast<double **>(&ctx->dgcount), (nk + 1) / 2});
    }
    size_t bytes = 0;
    auto al = [](size_t b) { return (b + 255) / 256 * 256; };
    for (auto &p : plan) bytes += al(sizeof(double) * p.second);
    bytes += al(sizeof(int) * 4);
    const size_t small = bytes;
    bytes += nf1 * mat;          // screening matrices / factors
    // Q (= Y), Z, P, Y', Z': real, or nk planar complex matrices for a periodic system
    const size_t matq = ctx->periodic ? mat * 2 * static_cast<size_t>(nk) : mat;
    bytes += 5 * matq;
    const int prec = ctx->opt.precision;
    // the mixed modes' iteration buffers: the matrix order, or the order of a cell's embedded
    // Hermitian matrices
    const long long ldm = ctx->periodic ? ctx->lde : ld;
    ctx->mgroup = groups && !ctx->lim.none && ctx->periodic && !fp64_path(prec) ? mixed_group(static_cast<int>(nk), ldm, prec) : 1;
    const size_t mat32 = sizeof(float) * static_cast<size_t>(ldm) * ldm * ctx->mgroup, mat16 = mat32 / 2;
    const size_t split_mat = prec == MBD_PREC_BF16X3 ? mat16 : (prec == MBD_PREC_TF32X3 ? mat32 : 0);
    if (!fp64_path(prec)) bytes += 6 * mat32;
    const size_t emat = sizeof(double) * static_cast<size_t>(ctx->lde) * ctx->lde * ctx->mgroup;
    const bool embed = ctx->periodic && !fp64_path(prec);
    if (embed) bytes += 5 * emat;
    bytes += 12 * split_mat;
    // FP32 screening factors, their diagonal-block inverses and solve workspace
    const size_t panel_words = 2 * nf1 * static_cast<size_t>(ld) * kScsPanel;
    const size_t grad32 = 2 * nf1 * (3 * static_cast<size_t>(ld) + N);
    const size_t scs32 = !fp64_path(prec) && !ctx->periodic   // cells screen in FP64 (Gamma point)
                             ? nf1 * (mat / 2) + al(sizeof(float) * nf1 * nb * 4096) +
                                   al(sizeof(float) * 2 * nf1 * ld * 3) + al(sizeof(uint32_t) * panel_words) +
                                   al(sizeof(float) * grad32)
                             : 0;
    bytes += scs32;
    // Scratch of the tensor-core products, taken only where it fits: FP64 products and factors (and the
    // transpose of P), and the build of Q(q), which can share theirs.
    const size_t q_work = ctx->periodic ? al(cell_products_bytes(ctx->N, ctx->cell, static_cast<int>(nk), ctx->maxG, prec, ctx->lim)) : 0;
    const size_t crt_part =
        fp64_path(prec) ? std::max({al(cholesky_crt_bytes(ld, static_cast<int>(nf1), ctx->lim)),
                                    al(ctx->periodic ? crt_cell_bytes(ctx->n, static_cast<int>(nk), ctx->lim) : crt_ns_bytes(ctx->n, ctx->lim)), q_work})
                        : q_work;
    const size_t pt_part = fp64_path(prec) ? matq : 0, crt_wanted = crt_part + pt_part;
    const size_t crt_work = ctx->lim.none ? 0 : crt_wanted;
    // A slab large enough for the new size is re-carved in place (systems of varying size in
    // a batch then reuse one allocation); otherwise it is replaced.
    cudaError_t e = cudaSuccess;
    if (!ctx->slab || ctx->slab_bytes < bytes + crt_work) {
        release(ctx);
        size_t want = bytes + crt_work;
        e = cudaMalloc(&ctx->slab, want);
        if (e != cudaSuccess && ctx->mgroup > 1) {   // one matrix at a time
            cudaGetLastError();
            ctx->slab = nullptr;
            return allocate(ctx, false);
        }
        if (e != cudaSuccess && crt_work) {   // without the tensor-core products' scratch
            cudaGetLastError();
            want = bytes;
            e = cudaMalloc(&ctx->slab, want);
        }
        if (e != cudaSuccess) {
            ctx->slab = nullptr;
            return cuda_fail(ctx, "mbd_set_geometry", e);
        }
        ctx->slab_bytes = want;
    }
    const bool crt = crt_work && ctx->slab_bytes >= bytes + crt_work;
    ctx->no_scratch = crt_wanted && !crt;
    ctx->qwork_bytes = crt ? q_work : 0;
    if (ctx->qslab) cudaFree(ctx->qslab);
    ctx->qslab = nullptr;
    char *scratch = crt ? static_cast<char *>(ctx->slab) + bytes + pt_part : nullptr;
    ctx->dPT = crt && pt_part ? reinterpret_cast<double *>(static_cast<char *>(ctx->slab) + bytes) : nullptr;
    ctx->crt = pt_part ? scratch : nullptr;
    ctx->qwork = q_work ? scratch : nullptr;
    char *p = static_cast<char *>(ctx->slab);
    for (auto &q : plan) {
        *q.first = reinterpret_cast<double *>(p);
        p += al(sizeof(double) * q.second);
    }
    ctx->dstatus = reinterpret_cast<int *>(p);
    p = static_cast<char *>(ctx->slab) + small;
    ctx->dM = reinterpret_cast<double *>(p);
    p += nf1 * mat;
    double **mats[5] = {&ctx->dQ, &ctx->dZ, &ctx->dP, &ctx->dY2, &ctx->dZ2};
    for (auto m : mats) {
        *m = reinterpret_cast<double *>(p);
        p += matq;
    }
    if (!fp64_path(prec)) {
        float **f32[6] = {&ctx->fY, &ctx->fZ, &ctx->fY2, &ctx->fZ2, &ctx->fP, &ctx->fPT};
        for (auto m : f32) {
            *m = reinterpret_cast<float *>(p);
            p += mat32;
        }
    }
    if (split_mat) {
        void **parts[6] = {ctx->hY, ctx->hZ, ctx->hY2, ctx->hZ2, ctx->hP, ctx->hPT};
        for (auto m : parts)
            for (int k = 0; k < 2; ++k) {
                m[k] = p;
                p += split_mat;
            }
    }
    if (embed) {
        double **em[5] = {&ctx->eM, &ctx->eV, &ctx->eW, &ctx->eVT, &ctx->eZ};
        for (auto m : em) {
            *m = reinterpret_cast<double *>(p);
            p += emat;
        }
    }
    if (scs32) {
        ctx->sM = reinterpret_cast<float *>(p);
        p += nf1 * (mat / 2);
        ctx->sdinv = reinterpret_cast<float *>(p);
        p += al(sizeof(float) * nf1 * nb * 4096);
        ctx->swork = reinterpret_cast<float *>(p);
        p += al(sizeof(float) * 2 * nf1 * ld * 3);
        ctx->spanel = reinterpret_cast<uint32_t *>(p);
        p += al(sizeof(uint32_t) * panel_words);
        ctx->sgrad32 = reinterpret_cast<float *>(p);
        p += al(sizeof(float) * grad32);
    }
    // Untouched parts of the factor buffers (strict upper triangles) are read by no
    // kernel; clearing them once keeps them finite.
    e = cudaMemset(ctx->slab, 0, bytes);
    if (e != cudaSuccess) return cuda_fail(ctx, "mbd_set_geometry", e);
    e = cudaMemcpy(ctx->du, ctx->hu.data(), sizeof(double) * nf1, cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(ctx->dwu, ctx->hwu.data(), sizeof(double) * nf1, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_fail(ctx, "mbd_set_geometry", e);
    return MBD_OK;
}

// Uploads the Bloch vectors and reciprocal-vector lists of a periodic geometry.
int upload_periodic(mbd_ctx *ctx) {
    cudaError_t e = cudaMemcpy(ctx->dkq, ctx->hkq.data(), sizeof(double) * ctx->hkq.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(ctx->dkw, ctx->hkw.data(), sizeof(double) * ctx->hkw.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(ctx->dG, ctx->hG.data(), sizeof(double) * ctx->hG.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(ctx->dglist, ctx->hglist.data(), sizeof(int) * ctx->hglist.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(ctx->dgcount, ctx->hgcount.data(), sizeof(int) * ctx->hgcount.size(), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_fail(ctx, "mbd_set_geometry", e);
    return MBD_OK;
}

PeriodicBufs periodic_bufs(mbd_ctx *ctx) {
    return PeriodicBufs{ctx->cell, ctx->nk, ctx->nkt, ctx->nG, ctx->maxG, ctx->dkq, ctx->dkw, ctx->dG, ctx->dglist, ctx->dgcount, ctx->dS};
}

// Host preparation of a periodic geometry: cell inverse and reciprocal vectors, Ewald
// parameters, Monkhorst-Pack Bloch vectors and the reciprocal vectors of each.
struct PeriodicSetup {
    CellGeom cell{};
    int nk = 0, nkt = 0, nG = 0, maxG = 0;
    std::vector<double> kq, kw, G;
    std::vector<int> glist, gcount;
    std::string msg;
};

int periodic_setup(const mbd_options &o, const double *A, const int *grid, PeriodicSetup &ps) {
    const double pi = 3.141592653589793238462643383279502884;
    for (int e = 0; e < 9; ++e)
        if (!std::isfinite(A[e])) { ps.msg = "non-finite lattice"; return MBD_ERR_INPUT; }
    for (int c = 0; c < 3; ++c)
        if (grid[c] < 1 || grid[c] > 64) { ps.msg = "k_grid entries must lie in 1..64"; return MBD_ERR_INPUT; }
    CellGeom &c = ps.cell;
    for (int e = 0; e < 9; ++e) c.A[e] = A[e];
    const double co[9] = {A[4] * A[8] - A[5] * A[7], -(A[3] * A[8] - A[5] * A[6]), A[3] * A[7] - A[4] * A[6],
                          -(A[1] * A[8] - A[2] * A[7]), A[0] * A[8] - A[2] * A[6], -(A[0] * A[7] - A[1] * A[6]),
                          A[1] * A[5] - A[2] * A[4], -(A[0] * A[5] - A[2] * A[3]), A[0] * A[4] - A[1] * A[3]};
    const double det = A[0] * co[0] + A[1] * co[1] + A[2] * co[2];
    if (!(std::fabs(det) > 1e-12)) { ps.msg = "singular lattice"; return MBD_ERR_INPUT; }
    for (int e = 0; e < 3; ++e)
        for (int k = 0; k < 3; ++k) c.Ainv[3 * e + k] = co[3 * k + e] / det;   // (A^{-1})_{ek}
    for (int k = 0; k < 3; ++k)
        for (int e = 0; e < 3; ++e) c.B[3 * k + e] = 2.0 * pi * c.Ainv[3 * e + k];
    c.vol = std::fabs(det);
    double g = o.ewald_gamma, rc = o.real_cutoff, kc = o.recip_cutoff;
    if (!(g > 0.0)) g = rc > 0.0 ? 6.0 / rc : 2.5 / std::cbrt(c.vol);
    if (!(rc > 0.0)) rc = 6.0 / g;
    if (!(kc > 0.0)) kc = 10.0 * g;
    c.gamma = g;
    c.rc = rc;
    c.kc = kc;
    auto norm = [](const double *v) { return std::sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]); };
    // Monkhorst-Pack: kappa_c = (2m - n_c - 1)/(2 n_c), q = kappa B.  The grid holds -q with every q, and
    // Q(-q) is the conjugate of Q(q), with the same spectrum and the conjugate inverse root: the FP64 path keeps
    // one of the two with weight 2.  (The mixed modes' rounding differs between the two; they keep
    // the whole grid.)
    const bool pairs = fp64_path(o.precision);
    ps.nkt = grid[0] * grid[1] * grid[2];
    double qmax = 0.0;
    for (int m0 = 1; m0 <= grid[0]; ++m0)
        for (int m1 = 1; m1 <= grid[1]; ++m1)
            for (int m2 = 1; m2 <= grid[2]; ++m2) {
                const int t[3] = {2 * m0 - grid[0] - 1, 2 * m1 - grid[1] - 1, 2 * m2 - grid[2] - 1};
                const int sign = t[0] ? t[0] : (t[1] ? t[1] : t[2]);
                if (pairs && sign < 0) continue;
                ps.kw.push_back(pairs && sign > 0 ? 2.0 : 1.0);
                const double kap[3] = {(2.0 * m0 - grid[0] - 1) / (2.0 * grid[0]),
                                       (2.0 * m1 - grid[1] - 1) / (2.0 * grid[1]),
                                       (2.0 * m2 - grid[2] - 1) / (2.0 * grid[2])};
                double q[3];
                for (int e = 0; e < 3; ++e) q[e] = kap[0] * c.B[e] + kap[1] * c.B[3 + e] + kap[2] * c.B[6 + e];
                for (int e = 0; e < 3; ++e) ps.kq.push_back(q[e]);
                qmax = std::max(qmax, norm(q));
            }
    ps.nk = static_cast<int>(ps.kw.size());
    // every G = m B with |G + q| < kc for some q: |G| < kc + qmax, |m_c| <= (kc + qmax)|a_c|/(2 pi)
    const double gr = kc + qmax;
    int mm[3];
    for (int k = 0; k < 3; ++k) mm[k] = static_cast<int>(std::floor(gr * norm(c.A + 3 * k) / (2.0 * pi))) + 1;
    const long long box = (2LL * mm[0] + 1) * (2LL * mm[1] + 1) * (2LL * mm[2] + 1);
    if (box > 20000000LL) { ps.msg = "reciprocal cutoff too large for this cell"; return MBD_ERR_INPUT; }
    for (int m0 = -mm[0]; m0 <= mm[0]; ++m0)
        for (int m1 = -mm[1]; m1 <= mm[1]; ++m1)
            for (int m2 = -mm[2]; m2 <= mm[2]; ++m2) {
                double G[3];
                for (int e = 0; e < 3; ++e) G[e] = m0 * c.B[e] + m1 * c.B[3 + e] + m2 * c.B[6 + e];
                if (norm(G) < gr) for (int e = 0; e < 3; ++e) ps.G.push_back(G[e]);
            }
    ps.nG = static_cast<int>(ps.G.size() / 3);
    std::vector<std::vector<int>> lists(ps.nk);
    for (int k = 0; k < ps.nk; ++k)
        for (int gi = 0; gi < ps.nG; ++gi) {
            double kv[3];
            for (int e = 0; e < 3; ++e) kv[e] = ps.G[3 * gi + e] + ps.kq[3 * k + e];
            const double kk = norm(kv);
            if (kk < kc && kk > 1e-12) lists[k].push_back(gi);
        }
    ps.maxG = 1;
    for (auto &l : lists) ps.maxG = std::max(ps.maxG, static_cast<int>(l.size()));
    ps.glist.assign(static_cast<size_t>(ps.nk) * ps.maxG, 0);
    ps.gcount.assign(ps.nk, 0);
    for (int k = 0; k < ps.nk; ++k) {
        ps.gcount[k] = static_cast<int>(lists[k].size());
        for (size_t t = 0; t < lists[k].size(); ++t) ps.glist[static_cast<size_t>(k) * ps.maxG + t] = lists[k][t];
    }
    if (ps.nG == 0) ps.nG = 1, ps.G.assign(3, 0.0);   // keeps the device arrays non-empty
    return MBD_OK;
}

struct Inputs {
    const double *R, *a0ref, *c6ref, *rref, *ratio;
};
struct Outputs {
    double *energy, *grad_coords, *grad_params, *alpha_scs;   // device pointers or null
};

AtomBufs atom_bufs(mbd_ctx *ctx, const Inputs &in) {
    return AtomBufs{ctx->N, ctx->nf1, in.R, in.a0ref, in.c6ref, in.rref, in.ratio,
                    ctx->da0, ctx->dom, ctx->drv, ctx->dalu, ctx->dsigu, ctx->dabar,
                    ctx->dabar0, ctx->dc6bar, ctx->dombar, ctx->drbar, ctx->du, ctx->dwu};
}

// Gradient passes (Sec. 2.4) from the state of the last forward evaluation: the MBD
// pair pass on Q^{-1/2}, the chain through the screened parameters, the adjoint solves
// V = A^{-1} H with the kept factors, the SCS pair pass and the TS chain.  Outputs are
// scaled by *grad_energy (device scalar) when it is given.
void backward_passes(mbd_ctx *ctx, cudaStream_t s, const AtomBufs &b, const double *grad_energy,
                     double *grad_coords, double *grad_params) {
    const long long ld = ctx->ld, mat = ld * ld, xs = 3 * ld;
    const double beta = ctx->opt.beta, a = ctx->opt.a;
    MbdGradOut go{ctx->dgomb, ctx->dgab0, ctx->dgrb, ctx->dgR};
    mbd_grad_pass(b, beta, a, ctx->Zlast, ld, ctx->zscale, go, s, ctx->tq_valid ? ctx->dtq : nullptr);
    if (ctx->opt.scs_mode == MBD_SCS_NL) {   // MBD-NL: only the chain through Eqs. mbd-nl-*
        if (grad_params) nl_chain(b, go, grad_energy, grad_params, s);
        if (grad_coords) scale_copy(ctx->dgR, 3 * ctx->N, grad_energy, grad_coords, s);
        return;
    }
    const bool fp64 = fp64_path(ctx->opt.precision);
    chain_screen(b, go, ctx->dh, ctx->dga0, ctx->dgrv, fp64 ? ctx->dV : ctx->dB, ld, xs, s);
    cudaMemsetAsync(ctx->dgom, 0, sizeof(double) * ctx->N, s);
    if (fp64)
        chol_solve3_f64(ctx->dM, ld, mat, ctx->nf1, ctx->ddinv, ctx->dV, ctx->dB, xs, s);
    else
        refine_solve3(ctx->dM, ctx->sM, ctx->sdinv, ld, ctx->n, ctx->nf1, ctx->dB, ctx->dV, ctx->swork,
                      kAdjointRefineSteps, s);
    scs_grad_pass(b, beta, a, ctx->dX, ctx->dV, xs, ctx->dga0, ctx->dgom, ctx->dgrv, ctx->dgR,
                  fp64 ? nullptr : ctx->sgrad32, ctx->dP, s);   // (P is free after the iteration)
    if (grad_params) ts_chain(b, ctx->dga0, ctx->dgom, ctx->dgrv, grad_energy, grad_params, s);
    if (grad_coords) scale_copy(ctx->dgR, 3 * ctx->N, grad_energy, grad_coords, s);
}

int read_status(mbd_ctx *ctx, cudaStream_t s, const char *origin) {
    int st = 0;
    MBD_CUDA(cudaMemcpyAsync(&st, ctx->dstatus, sizeof(int), cudaMemcpyDeviceToHost, s), origin);
    MBD_CUDA(cudaStreamSynchronize(s), origin);
    MBD_CUDA(cudaGetLastError(), origin);
    if (st & ST_INPUT) return fail(ctx, MBD_ERR_INPUT, origin, "non-finite or non-positive input, or coincident atoms");
    if (st & ST_TC_TIMEOUT) return fail(ctx, MBD_ERR_CUDA, origin, "tensor-core GEMM wait timed out");
    if (st & ST_SCS_NOT_PD)
        return fail(ctx, MBD_ERR_SCS_NOT_PD, origin, "screening matrix alpha^-1 + T^scs is not positive definite");
    if (st & ST_NEG_ALPHA)
        return fail(ctx, MBD_ERR_SCS_NEG_ALPHA, origin, "screened static polarizability or C6 is not positive");
    return MBD_OK;
}


// Operand set of one matrix in the mixed modes: FP32 values and, for BF16x3, hi/lo.
struct MixMat {
    float *f;
    void *h, *l;
    const void *op0(bool split) const { return split ? static_cast<const void *>(h) : static_cast<const void *>(f); }
    const void *op1(bool split) const { return split ? static_cast<const void *>(l) : static_cast<const void *>(f); }
};

// The matrices of a mixed-precision matrix function and where its results go: `count` of Q (FP64,
// symmetric, ld x ld, valid n x n, decoupled padding) one after another, the FP64 workspaces V, W and VT (ld^2
// doubles each a matrix), the FP64 outputs Zd ~ Q^{-1/2}, the energies [count], and (if tq is not NULL) for each
// the traces of the first N diagonal 3x3 blocks of Q^{1/2}, second order in the error of Zd.
struct MixProblem {
    const double *Q;
    long long ld;
    int n;
    double *V, *W, *VT, *Zd;
    double *tq, *energy;
    int count = 1;
};
// A matrix's scale and spectrum bounds (inputs), and how its iteration went.
struct MixItem {
    double sc, lbound, ubound;
    double resid = 0.0, prev = 1e300;
    int it = 0, code = MBD_OK;
    bool done = false;
    const float *Z = nullptr;   // its Z after the last step
};

// Mixed-precision coupled Newton-Schulz (same scaled steps as the FP64 loop) on the
// tensor cores, stopped at the precision floor, then the FP64 correction:
// Zd = Z/sqrt(s) ~ Q^{-1/2}, V = Q Zd, W = Zd V, E = (3 Tr V - sum V o W)/4 - 3/2 sum w.
// The FP32 and split-part buffers of the context hold the iteration (ld^2 elements each a matrix).
// The matrices of a group share launches and read-backs; each takes its own steps, as if it were alone, and
// leaves the group when it is done.
int newton_schulz_mixed(mbd_ctx *ctx, cudaStream_t s, const MixProblem &pr, std::vector<MixItem> &items,
                        std::vector<Span> &spans, cudaEvent_t &e_corr) {
    const long long ld = pr.ld, mat = ld * ld;
    const int n = pr.n, N = ctx->N, M = static_cast<int>(ld), count = pr.count;
    const int kind = ctx->opt.precision == MBD_PREC_TF32 ? 0 : (ctx->opt.precision == MBD_PREC_BF16X3 ? 1 : 2);
    const bool split = kind != 0;
    const double nd = static_cast<double>(n);
    const double flops_full = 2.0 * nd * nd * nd, flops_sym = nd * nd * (nd + 1.0);
    MixMat Y{ctx->fY, ctx->hY[0], ctx->hY[1]}, Z{ctx->fZ, ctx->hZ[0], ctx->hZ[1]};
    MixMat Y2{ctx->fY2, ctx->hY2[0], ctx->hY2[1]}, Z2{ctx->fZ2, ctx->hZ2[0], ctx->hZ2[1]};
    MixMat P{ctx->fP, ctx->hP[0], ctx->hP[1]}, PT{ctx->fPT, ctx->hPT[0], ctx->hPT[1]};
    auto at = [&](const MixMat &m, int k) {   // matrix k of the group
        const long long part = k * mat * (kind == 1 ? 2 : 4);
        auto moved = [&](void *p) { return split ? static_cast<void *>(static_cast<char *>(p) + part) : p; };
        return MixMat{m.f + k * mat, moved(m.h), moved(m.l)};
    };
    for (int k = 0; k < count; ++k) {
        const MixMat y = at(Y, k), z = at(Z, k);
        mixed_init(kind, pr.Q + k * mat, ld, 1.0 / items[k].sc, y.f, split ? y.h : nullptr, y.l, z.f, z.h, z.l, s);
    }
    // K stages per tensor-memory accumulation: the option, or the kind's default (BF16x3: 8,
    // i.e. 512 products per FP32 sum in tensor memory; TF32 and TF32x3: 2, i.e. 64 products)
    const int cstages = ctx->opt.tc_chunk_stages > 0 ? ctx->opt.tc_chunk_stages : (kind == 1 ? 8 : 2);
    // the correction's TF32x3 products keep short accumulations whatever the iteration's kind
    constexpr int kCorrectionChunk = 2;
    std::vector<int> active;   // matrices still iterated on
    for (int k = 0; k < count; ++k) active.push_back(k);
    // One product of every active matrix, timed; alpha and beta by matrix.
    auto tc = [&](int tk, const TcOperands &op, TcArgs g, double flops, const char *origin, auto alpha, auto beta) -> int {
        if (count == 1) {
            g.alpha = static_cast<float>(alpha(0));
            g.beta = static_cast<float>(beta(0));
        } else {
            g.batch = g.nslots = static_cast<int>(active.size());
            g.sC = mat;
            for (int j = 0; j < g.nslots; ++j) {
                g.slot[j] = active[j];
                g.alphas[j] = static_cast<float>(alpha(active[j]));
                g.betas[j] = static_cast<float>(beta(active[j]));
            }
        }
        Span sp;
        sp.flops = flops * static_cast<double>(active.size());
        mark(ctx, s, sp.a);
        const cudaError_t e = tc_gemm(tk, op, g, s);
        mark(ctx, s, sp.b);
        if (ctx->profiling) spans.push_back(sp);
        return e == cudaSuccess ? MBD_OK : cuda_fail(ctx, origin, e);
    };
    auto one = [](int) { return 1.0; };
    auto zero = [](int) { return 0.0; };
    double *resid_dev = ctx->dmix, *corr_dev = ctx->dmix + kTcSlots;
    std::vector<ns::Coeffs> cf(count);
    auto c1 = [&](int k) { return cf[k].c1; };
    auto c3 = [&](int k) { return cf[k].c3; };
    for (int it = 0; it < ctx->opt.ns_max_iter && !active.empty(); ++it) {
        MixMat Pk = Y, PTk = Y;   // P_0 = Y_0 (symmetric)
        if (it > 0) {
            MBD_CUDA(cudaMemsetAsync(resid_dev, 0, sizeof(double) * count, s), "newton_schulz_tc");
            TcOperands op{Z.op0(split), Z.op1(split), Y.op0(split), Y.op1(split), ld, ld};
            TcArgs g{M, M, M, 1.f, 0.f, nullptr, ld, split ? nullptr : P.f, split ? P.h : nullptr,
                     split ? P.l : nullptr, split ? nullptr : PT.f, split ? PT.h : nullptr, split ? PT.l : nullptr,
                     resid_dev, n, 0, ctx->dstatus};
            g.chunk_stages = cstages;
            // P = Z Y (and its transpose), resid = |I - P|_F^2
            if (const int rc = tc(kind, op, g, flops_full, "newton_schulz_tc", one, zero)) return rc;
            Pk = P;
            PTk = PT;
            double r2[kTcSlots] = {};
            MBD_CUDA(cudaMemcpyAsync(r2, resid_dev, sizeof(double) * count, cudaMemcpyDeviceToHost, s), "newton_schulz_tc");
            MBD_CUDA(cudaStreamSynchronize(s), "newton_schulz_tc");
            std::vector<int> good;
            for (int k : active) {
                MixItem &m = items[k];
                m.resid = std::sqrt(r2[k]);
                if (!std::isfinite(m.resid) || m.resid > 2.0 * std::sqrt(nd) + 1.0) {
                    m.it = it;
                    m.code = MBD_ERR_NEG_EIGENVALUE;
                } else {
                    good.push_back(k);
                }
            }
            active = good;
            if (active.empty()) break;
        }
        for (int k : active) {
            MixItem &m = items[k];
            // The tensor-core phase ends at its precision floor (ns::mixed_last).
            m.done = it > 0 && ns::mixed_last(m.resid, m.prev, ctx->opt.ns_tol, kMixedFloor * std::sqrt(nd));
            cf[k] = ns::step(m.lbound, m.ubound, m.done);
        }
        {   // Y' = c1 Y + c3 Y P = NT(Y, P^T): symmetric
            TcOperands op{Y.op0(split), Y.op1(split), PTk.op0(split), PTk.op1(split), ld, ld};
            TcArgs g{M, M, M, 0.f, 0.f, Y.f, ld, Y2.f, split ? Y2.h : nullptr, split ? Y2.l : nullptr, nullptr, nullptr,
                     nullptr, nullptr, 0, 2, ctx->dstatus};
            g.chunk_stages = cstages;
            if (const int rc = tc(kind, op, g, flops_sym, "newton_schulz_tc", c3, c1)) return rc;
        }
        if (it == 0) {
            for (int k : active) {
                const MixMat z = at(Z2, k);
                mixed_axpby_identity(kind, at(Y, k).f, ld, static_cast<float>(cf[k].c1), static_cast<float>(cf[k].c3), z.f,
                                     split ? z.h : nullptr, z.l, s);
            }
        } else {   // Z' = c1 Z + c3 P Z = NT(P, Z): symmetric
            TcOperands op{Pk.op0(split), Pk.op1(split), Z.op0(split), Z.op1(split), ld, ld};
            TcArgs g{M, M, M, 0.f, 0.f, Z.f, ld, Z2.f, split ? Z2.h : nullptr, split ? Z2.l : nullptr, nullptr, nullptr,
                     nullptr, nullptr, 0, 2, ctx->dstatus};
            g.chunk_stages = cstages;
            if (const int rc = tc(kind, op, g, flops_sym, "newton_schulz_tc", c3, c1)) return rc;
        }
        std::swap(Y, Y2);
        std::swap(Z, Z2);
        std::vector<int> left;
        for (int k : active) {
            MixItem &m = items[k];
            m.it = it + 1;
            if (it > 0) m.prev = m.resid;
            if (m.done) m.Z = Z.f + k * mat;
            else left.push_back(k);
        }
        active = left;
    }
    int st = 0;
    MBD_CUDA(cudaMemcpyAsync(&st, ctx->dstatus, sizeof(int), cudaMemcpyDeviceToHost, s), "newton_schulz_tc");
    MBD_CUDA(cudaStreamSynchronize(s), "newton_schulz_tc");
    if (st & ST_TC_TIMEOUT) return fail(ctx, MBD_ERR_CUDA, "newton_schulz_tc", "tensor-core GEMM wait timed out");
    active.clear();   // the matrices before the first one that failed
    for (int k = 0; k < count && items[k].done && items[k].code == MBD_OK; ++k) active.push_back(k);
    // ---- correction ----
    // With Zs ~ (Q/s)^{-1/2} (FP32 values of the iteration), Vs = (Q/s) Zs, Ws = Zs Vs:
    // Tr Q^{1/2} ~ sqrt(s) (3 Tr Vs - sum Vs o Ws)/2, second order in the error of Zs.
    // Tr Vs = sum (Q/s) o Zs is an exact FP64 dot.  Vs and Ws are FP64 sums of exact
    // diagonal scalings and TF32x3 tensor-core products of the off-diagonal parts (no
    // accumulator mixes a dominant term with many small ones; chunk sums in FP32 with
    // round-to-nearest), each product added once into its FP64 result.
    double c2[kTcSlots] = {};
    if (!active.empty()) {
        mark(ctx, s, e_corr);
        // FP32 workspace: the iteration's matrices other than Z are free now.  Parts of offdiag(Q/s) and of
        // the full Zs feed the first product; offdiag(Zs) (reusing the Q parts) and Vs^T the
        // second.
        float *Qh = Y.f, *Ql = Y2.f, *Zs_h = P.f, *Zs_l = PT.f, *Zh = Qh, *Zl = Ql;
        float *VTh = reinterpret_cast<float *>(pr.VT), *VTl = VTh + count * mat;
        for (int k : active) {
            const long long o = k * mat;
            split_tf32_f64(pr.Q + o, ld, 1.0 / items[k].sc, 1, Qh + o, Ql + o, s);
            split_tf32_f32(items[k].Z, ld, 0, Zs_h + o, Zs_l + o, s);
            diag_scale_rows_f64(pr.Q + o, items[k].Z, ld, 1.0 / items[k].sc, pr.V + o, s);
        }
        {   // Vs += offdiag(Q/s) Zs = NT(offdiag(Q/s), Zs) (Zs symmetric)
            TcOperands op{Qh, Ql, Zs_h, Zs_l, ld, ld};
            TcArgs g{M, M, M, 1.f, 0.f, nullptr, ld, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr,
                     0, 0, ctx->dstatus, pr.V, kCorrectionChunk};
            if (const int rc = tc(2, op, g, flops_full, "correction", one, zero)) return rc;
        }
        for (int k : active) {
            const long long o = k * mat;
            split_tf32_f64_t(pr.V + o, ld, 1.0, VTh + o, VTl + o, s);
            split_tf32_f32(items[k].Z, ld, 1, Zh + o, Zl + o, s);
            diag_scale_rows_f32(items[k].Z, pr.V + o, ld, pr.W + o, s);
        }
        {   // Ws += offdiag(Zs) Vs = NT(offdiag(Zs), Vs^T)
            TcOperands op{Zh, Zl, VTh, VTl, ld, ld};
            TcArgs g{M, M, M, 1.f, 0.f, nullptr, ld, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr,
                     0, 0, ctx->dstatus, pr.W, kCorrectionChunk};
            if (const int rc = tc(2, op, g, flops_full, "correction", one, zero)) return rc;
        }
        for (int k : active) {
            const long long o = k * mat;
            const double sc = items[k].sc;
            energy_correction(pr.Q + o, 1.0 / sc, items[k].Z, pr.V + o, pr.W + o, ld, n, std::sqrt(sc), ctx->dombar, N,
                              ctx->dscal + 8 + 2 * 64, pr.energy + k, corr_dev + k, s);
            if (pr.tq)   // diagonal blocks of Q^{1/2}, second order in the error of Zs, for dE/d omega_bar
                block_trace_sqrt(pr.V + o, pr.W + o, ld, N, std::sqrt(sc), pr.tq + static_cast<long long>(k) * N, s);
            to_f64(items[k].Z, ld, 1.0 / std::sqrt(sc), pr.Zd + o, s);   // Q^{-1/2} for the gradient
        }
        MBD_CUDA(cudaMemcpyAsync(c2, corr_dev, sizeof(double) * count, cudaMemcpyDeviceToHost, s), "correction");
        int st2 = 0;
        MBD_CUDA(cudaMemcpyAsync(&st2, ctx->dstatus, sizeof(int), cudaMemcpyDeviceToHost, s), "correction");
        MBD_CUDA(cudaStreamSynchronize(s), "correction");
        if (st2 & ST_TC_TIMEOUT) return fail(ctx, MBD_ERR_CUDA, "correction", "tensor-core GEMM wait timed out");
    }
    for (int k = 0; k < count; ++k) {
        const MixItem &m = items[k];
        ctx->ns_iter = m.it;
        ctx->ns_resid = m.resid;
        if (m.code != MBD_OK)
            return fail(ctx, m.code, "newton_schulz_tc", "Q has a non-positive eigenvalue (polarization catastrophe)");
        if (!m.done) return fail(ctx, MBD_ERR_NOT_CONVERGED, "newton_schulz_tc", "iteration cap reached");
        ctx->corr_resid = k ? std::max(ctx->corr_resid, c2[k]) : c2[k];
        // The corrected energy is second order in the error of Zs: with Zs = (Q/s)^{-1/2} (I + F),
        // Ws - I ~ 2F and the error of Tr Q^{1/2}/2 is about (3/4) Tr(Q^{1/2} F^2) <= (3/16) sqrt(s) r^2.
        // The split kinds claim the 1e-6 Ha/atom bar; a Z too poor for it is reported, not used.
        if (split && !(3.0 / 16.0 * std::sqrt(m.sc) * c2[k] * c2[k] / (n / 3) <= ctx->opt.mixed_max_error))
            return fail(ctx, MBD_ERR_NOT_CONVERGED, "correction",
                        "the tensor-core Q^{-1/2} is too inaccurate for the energy bar (mixed_max_error)");
    }
    ctx->Zlast = pr.Zd;
    ctx->zscale = 1.0;
    return MBD_OK;
}

// Gradient passes of a periodic system: the MBD pair pass over Bloch vectors (atoms,
// screened parameters, lattice), the chain through the screened parameters, the adjoint
// solves on the Gamma-point factors and the SCS pass over lattice images.
int backward_periodic(mbd_ctx *ctx, cudaStream_t s, const AtomBufs &b, const double *grad_energy,
                      double *grad_coords, double *grad_params) {
    const long long ld = ctx->ld, mat = ld * ld, xs = 3 * ld;
    const double beta = ctx->opt.beta, a = ctx->opt.a;
    const PeriodicBufs pb = periodic_bufs(ctx);
    MbdGradOut go{ctx->dgomb, ctx->dgab0, ctx->dgrb, ctx->dgR};
    const bool mixed = ctx->opt.precision != MBD_PREC_FP64 && ctx->opt.precision != MBD_PREC_FP64_SPLIT;
    const size_t bytes = grad_products_bytes(ctx->N, ctx->cell, ctx->nk, ctx->maxG, ctx->lim);
    char *products = ctx->qwork && bytes && bytes <= ctx->qwork_bytes ? ctx->qwork : nullptr;
    if (products) MBD_CUDA(cudaMemsetAsync(ctx->dstatus, 0, sizeof(int), s), "gradient");
    MBD_CUDA(periodic_mbd_grad(b, pb, beta, a, ctx->Zlast, ld, ctx->zscale, go, ctx->dgc, ctx->dgA, s,
                               ctx->tq_valid ? ctx->dtq : nullptr, mixed, products, ctx->dstatus, ctx->lim), "gradient");
    if (ctx->opt.scs_mode == MBD_SCS_NL) {   // MBD-NL: no screening to differentiate
        if (grad_params) nl_chain(b, go, grad_energy, grad_params, s);
        if (grad_coords) scale_copy(ctx->dgR, 3 * ctx->N, grad_energy, grad_coords, s);
        scale_copy(ctx->dgA, 9, grad_energy, ctx->dgAout, s);
        if (products) {   // its tensor-core waits are bounded: check them
            if (const int rc = read_status(ctx, s, "gradient")) return rc;
        }
        ctx->have_lattice_grad = true;
        return MBD_OK;
    }
    chain_screen(b, go, ctx->dh, ctx->dga0, ctx->dgrv, ctx->dV, ld, xs, s);
    cudaMemsetAsync(ctx->dgom, 0, sizeof(double) * ctx->N, s);
    chol_solve3_f64(ctx->dM, ld, mat, ctx->nf1, ctx->ddinv, ctx->dV, ctx->dB, xs, s);
    scs_grad_periodic(b, ctx->cell, beta, a, ctx->dX, ctx->dV, xs, ctx->dga0, ctx->dgom, ctx->dgrv, ctx->dgR,
                      ctx->dgApart, ctx->dgA, s);
    if (grad_params) ts_chain(b, ctx->dga0, ctx->dgom, ctx->dgrv, grad_energy, grad_params, s);
    if (grad_coords) scale_copy(ctx->dgR, 3 * ctx->N, grad_energy, grad_coords, s);
    scale_copy(ctx->dgA, 9, grad_energy, ctx->dgAout, s);
    if (products) {
        if (const int rc = read_status(ctx, s, "gradient")) return rc;
    }
    ctx->have_lattice_grad = true;
    return MBD_OK;
}

// Periodic evaluation (Secs. 2.2 and 2.3): Gamma-point screening, Q(q) for the Bloch vectors of the grid, batched
// complex coupled Newton-Schulz (FP64: each complex product as one real product of residues, or as 4 real GEMMs on the
// FP64 pipe where the scratch does not fit; the tensor-core modes take each Q(q) as its real symmetric embedding
// through the finite matrix function), E = (1/nkt) sum_q kw_q 1/2 Tr Q(q)^{1/2} - 3/2 sum omega_bar.
int run_periodic(mbd_ctx *ctx, cudaStream_t s, const Inputs &in, const Outputs &out, bool want_grad) {
    if (ctx->opt.scs_mode == MBD_SCS_LEARNED)
        return fail(ctx, MBD_ERR_UNSUPPORTED, "learned_screening", "learned screening is for finite systems");
    const int N = ctx->N, n = ctx->n, nf1 = ctx->nf1, nk = ctx->nk;
    const long long ld = ctx->ld, mat = ld * ld, xs = 3 * ld;
    const double beta = ctx->opt.beta, a = ctx->opt.a;
    ctx->have_result = false;
    ctx->have_screening = false;
    ctx->have_forward = false;
    ctx->have_lattice_grad = false;
    ctx->tq_valid = false;
    ctx->ev_used = 0;
    ctx->prof = mbd_profile{};
    const long long launches0 = launch_count();
    cudaEvent_t e_start = nullptr, e_scs = nullptr, e_ns = nullptr, e_grad = nullptr;
    std::vector<Span> gemms;
    const double nd = static_cast<double>(n);
    const double flops_cplx = 8.0 * nd * nd * nd * nk;   // one complex product per Bloch vector
    cudaError_t crt_err = cudaSuccess;   // first launch error of the tensor-core products
    // herm: Hermitian result, of which one triangle is formed (about half the work on the FP64 pipe).
    // Bt, conj: the rows of B^T for the tensor cores; T: also the transpose (there only).
    auto timed_cgemm = [&](const double *A, const double *B, const double *Bt, bool conj, const double *D, double *C,
                           double *T, double alpha, double bt, bool herm) {
        Span sp;
        sp.flops = herm ? 4.0 * nd * nd * (nd + 1.0) * nk : flops_cplx;
        mark(ctx, s, sp.a);
        if (ctx->crt) {
            const cudaError_t e = crt_cell_product(ctx, A, Bt, conj, D, C, T, alpha, bt, herm, s);
            if (crt_err == cudaSuccess) crt_err = e;
        } else {
            cgemm_f64(A, B, D, C, ld, nk, alpha, bt, herm, s);
        }
        mark(ctx, s, sp.b);
        if (ctx->profiling) gemms.push_back(sp);
    };
    const AtomBufs b = atom_bufs(ctx, in);
    const PeriodicBufs pb = periodic_bufs(ctx);
    NvtxStages nv;
    nv.next("mbd screening (periodic)");
    mark(ctx, s, e_start);
    MBD_CUDA(cudaMemsetAsync(ctx->dstatus, 0, sizeof(int), s), "mbd_evaluate");
    // ---- Gamma-point screening (MBD-NL: the oscillators directly) ----
    if (ctx->opt.scs_mode == MBD_SCS_NL) {
        nl_params(b, ctx->dstatus, s);
        structure_factors(b, pb, s);
    } else {
        prepare_atoms(b, ctx->dstatus, s);
        structure_factors(b, pb, s);
        build_scs_periodic(b, ctx->cell, beta, a, ctx->dM, ld, mat, ctx->dstatus, s);
        if (const int rf = factorise(ctx, ctx->dM, nf1, s, "screening")) return rf;
        init_rhs_identity(ctx->dX, ld, n, nf1, xs, s);
        chol_solve3_f64(ctx->dM, ld, mat, nf1, ctx->ddinv, ctx->dX, ctx->dB, xs, s);
        contract_screen(b, ctx->dX, ld, xs, ctx->dstatus, s);
    }
    mark(ctx, s, e_scs);
    nv.next("mbd coupled oscillators and Newton-Schulz");
    int rc = read_status(ctx, s, "screening");
    if (rc) return rc;
    ctx->have_screening = true;
    // ---- Q(q) and the spectrum bounds ----
    const size_t qbytes = build_q_products_bytes(N, ctx->cell, nk, ctx->maxG, ctx->lim);
    if (fp64_path(ctx->opt.precision) && ctx->qwork && qbytes && qbytes <= ctx->qwork_bytes) {
        MBD_CUDA(build_q_products(b, pb, beta, a, ctx->dQ, ld, ctx->qwork, ctx->dstatus, s, ctx->lim), "coupled_oscillator_matrix");
        pad_q_periodic(b, pb, ctx->dQ, ld, n, s);
    } else {
        build_q_periodic(b, pb, beta, a, ctx->dQ, ld, n, ctx->dstatus, s);
    }
    cmax_abs_rowsum(ctx->dQ, ld, nk, ctx->dscal + 1, s);
    double sc = 0.0;
    MBD_CUDA(cudaMemcpyAsync(&sc, ctx->dscal + 1, sizeof(double), cudaMemcpyDeviceToHost, s), "newton_schulz");
    rc = read_status(ctx, s, "coupled_oscillator_matrix");
    if (rc) return rc;
    if (!(sc > 0.0) || !std::isfinite(sc)) return fail(ctx, MBD_ERR_INPUT, "newton_schulz", "invalid Q scale");
    double *energy_out = out.energy ? out.energy : ctx->dscal;
    std::vector<Span> tc_spans;
    if (!fp64_path(ctx->opt.precision)) {
        // ---- mixed modes: each Hermitian Q(q) as its real symmetric embedding [[Re, -Im],
        // [Im, Re]] (the same spectrum, twice) through the finite mixed-precision matrix function:
        // tensor-core iteration with its own scale and bounds, FP64 correction of the energy ----
        cudaEvent_t e_corr = nullptr;
        const long long lde = ctx->lde;
        const int ne = 2 * n, lzs = std::min(kLanczosSteps, static_cast<int>(lde));
        int it_max = 0;
        double res_max = 0.0, corr_max = 0.0, sc_max = 0.0;
        std::vector<double> lzk;
        double *energies = ctx->dcoef + static_cast<long long>(nk) * 2 * kLanczosSteps;
        double *rowsum = ctx->dmix + 2 * kTcSlots;
        const long long emat = lde * lde;
        for (int k0 = 0; k0 < nk; k0 += ctx->mgroup) {
            const int g = std::min(ctx->mgroup, nk - k0);
            for (int k = 0; k < g; ++k) {
                embed_hermitian(ctx->dQ, ld, n, k0 + k, ctx->eM + k * emat, lde, s);
                max_abs_rowsum(ctx->eM + k * emat, lde, static_cast<int>(lde), rowsum + k, s);
            }
            double sums[kTcSlots] = {};
            MBD_CUDA(cudaMemcpyAsync(sums, rowsum, sizeof(double) * g, cudaMemcpyDeviceToHost, s), "newton_schulz");
            lanczos_coefficients_f32(ctx->eM, ctx->fY, lde, lzs, ctx->eV, ctx->dcoef, s, g, emat);
            lzk.resize(static_cast<size_t>(g) * 2 * lzs);
            MBD_CUDA(cudaMemcpyAsync(lzk.data(), ctx->dcoef, sizeof(double) * lzk.size(), cudaMemcpyDeviceToHost, s),
                     "newton_schulz");
            MBD_CUDA(cudaStreamSynchronize(s), "newton_schulz");
            std::vector<MixItem> items(g);
            for (int k = 0; k < g; ++k) {
                double sk = sums[k];
                if (!(sk > 0.0) || !std::isfinite(sk))
                    return fail(ctx, MBD_ERR_INPUT, "newton_schulz", "invalid Q scale");
                double lo = 0.0, hi = sk;
                const double *lz = lzk.data() + static_cast<size_t>(k) * 2 * lzs;
                std::vector<double> da, db;
                for (int j = 0; j < lzs; ++j) {
                    da.push_back(lz[2 * j]);
                    if (j + 1 < lzs) db.push_back(lz[2 * j + 1]);
                    if (!(lz[2 * j + 1] > 1e-14 * sk)) break;
                }
                db.resize(da.empty() ? 0 : da.size() - 1);
                if (!da.empty()) tridiag_extremes(da, db, lo, hi);
                double ub = 1.0;
                if (std::isfinite(hi) && hi > 0.0 && 1.05 * hi < sk) {
                    sk = 1.05 * hi;
                    ub = 1.05;
                }
                items[k].sc = sk;
                items[k].lbound = ns::lower_estimate(lo, sk);   // an estimate (ns_schedule.h)
                items[k].ubound = ub;
            }
            // Re Tr (Q(q_k)^{1/2})_ii: the first N diagonal blocks of M_k^{1/2}, into row k of dlzw
            const MixProblem pr{ctx->eM, lde, ne, ctx->eV, ctx->eW, ctx->eVT, ctx->eZ,
                                ctx->dlzw + static_cast<long long>(k0) * N, energies + k0, g};
            const int rk = newton_schulz_mixed(ctx, s, pr, items, tc_spans, e_corr);
            if (rk) return rk;
            for (int k = 0; k < g; ++k) extract_hermitian(ctx->eZ + k * emat, lde, n, ctx->dZ, ld, k0 + k, s);
            for (const MixItem &m : items) {
                it_max = std::max(it_max, m.it);
                res_max = std::max(res_max, m.resid);
                sc_max = std::max(sc_max, m.sc);
            }
            corr_max = std::max(corr_max, ctx->corr_resid);
        }
        ctx->ns_iter = it_max;
        ctx->ns_resid = res_max;
        ctx->corr_resid = corr_max;
        ctx->ns_scale = sc_max;
        periodic_mixed_energy(energies, nk, ctx->dombar, N, energy_out, s);
        mean_rows(ctx->dlzw, nk, N, ctx->dtq, s);   // (1/nk) sum_q Re Tr (Q(q)^{1/2})_ii
        ctx->tq_valid = true;
        ctx->Zlast = ctx->dZ;
        ctx->zscale = 1.0;
    } else {
    const int lz_steps = std::min(kLanczosSteps, static_cast<int>(2 * ld));
    clanczos_coefficients(ctx->dQ, ld, nk, lz_steps, ctx->dlzw, ctx->dcoef, s);
    std::vector<double> lz(static_cast<size_t>(nk) * 2 * lz_steps);
    MBD_CUDA(cudaMemcpyAsync(lz.data(), ctx->dcoef, sizeof(double) * lz.size(), cudaMemcpyDeviceToHost, s),
             "newton_schulz");
    MBD_CUDA(cudaStreamSynchronize(s), "newton_schulz");
    double th_min = 1e300, th_max = 0.0;
    for (int k = 0; k < nk; ++k) {
        std::vector<double> da, db;
        const double *c = lz.data() + static_cast<size_t>(k) * 2 * lz_steps;
        for (int j = 0; j < lz_steps; ++j) {
            da.push_back(c[2 * j]);
            if (!(c[2 * j + 1] > 1e-14 * sc)) break;
            if (j + 1 < lz_steps) db.push_back(c[2 * j + 1]);
        }
        db.resize(da.empty() ? 0 : da.size() - 1);
        double lo = 0.0, hi = sc;
        if (!da.empty()) tridiag_extremes(da, db, lo, hi);
        th_min = std::min(th_min, lo);
        th_max = std::max(th_max, hi);
    }
    double ubound = 1.0;
    if (std::isfinite(th_max) && th_max > 0.0 && 1.05 * th_max < sc) {
        sc = 1.05 * th_max;
        ubound = 1.05;
    }
    ctx->ns_scale = sc;
    // the smallest over all Bloch vectors; an estimate, which may lie above the true bound
    // (that costs steps only, ns_schedule.h)
    double lbound = ns::lower_estimate(th_min, sc, 0.5);
    const double ss = std::sqrt(sc);
    // ---- batched complex coupled Newton-Schulz (same scaled steps as the finite path) ----
    double *Y = ctx->dQ, *Z = ctx->dZ, *P = ctx->dP, *Y2 = ctx->dY2, *Z2 = ctx->dZ2;
    cscale(Y, ld, nk, 1.0 / sc, s);
    cset_identity(Z, ld, nk, s);
    bool converged = false;
    double resid = 0.0;
    int it = 0;
    for (; it < ctx->opt.ns_max_iter; ++it) {
        const double *Pk = Y;
        if (it > 0) {
            timed_cgemm(Z, Y, Y, true, nullptr, P, ctx->dPT, 1.0, 0.0, false);   // P = Z Y: not Hermitian in floating point
            Pk = P;
        }
        cfrob_dev_identity(Pk, ld, n, nk, ctx->dkw, ctx->dscal + 2, s);
        double r2 = 0.0;
        MBD_CUDA(cudaMemcpyAsync(&r2, ctx->dscal + 2, sizeof(double), cudaMemcpyDeviceToHost, s), "newton_schulz");
        MBD_CUDA(cudaStreamSynchronize(s), "newton_schulz");
        resid = std::sqrt(r2);
        if (!std::isfinite(resid) || resid > 2.0 * std::sqrt(nd * ctx->nkt) + 1.0) {
            ctx->ns_iter = it;
            ctx->ns_resid = resid;
            return fail(ctx, MBD_ERR_NEG_EIGENVALUE, "newton_schulz",
                        "Q(q) has a non-positive eigenvalue (polarization catastrophe)");
        }
        const bool last = resid < ctx->opt.ns_tol;
        const ns::Coeffs cf = ns::step(lbound, ubound, last);
        const double c1 = cf.c1, c3 = cf.c3;
        // Y' = c1 Y + c3 Y P (Hermitian: Y Z Y; P_0 = Y_0)
        timed_cgemm(Y, Pk, it == 0 ? Y : ctx->dPT, it == 0, Y, Y2, nullptr, c3, c1, kHermitianNs);
        if (it == 0) caxpby_identity(Z2, Pk, ld, nk, c1, c3, s);
        else timed_cgemm(Pk, Z, Z, true, Z, Z2, nullptr, c3, c1, kHermitianNs);   // Z' = c1 Z + c3 P Z (Hermitian: Z Y Z)
        if (crt_err != cudaSuccess) return cuda_fail(ctx, "newton_schulz", crt_err);
        std::swap(Y, Y2);
        std::swap(Z, Z2);
        if (last) {
            converged = true;
            ++it;
            break;
        }
    }
    ctx->ns_iter = it;
    ctx->ns_resid = resid;
    if (ctx->crt) {   // tensor-core waits are bounded: check them
        int st = 0;
        MBD_CUDA(cudaMemcpyAsync(&st, ctx->dstatus, sizeof(int), cudaMemcpyDeviceToHost, s), "newton_schulz");
        MBD_CUDA(cudaStreamSynchronize(s), "newton_schulz");
        if (st & ST_TC_TIMEOUT) return fail(ctx, MBD_ERR_CUDA, "newton_schulz", "tensor-core GEMM wait timed out");
    }
    if (!converged) return fail(ctx, MBD_ERR_NOT_CONVERGED, "newton_schulz", "iteration cap reached");
    energy_trace_periodic(Y, ld, n, periodic_bufs(ctx), ctx->dombar, N, ss, energy_out, s);
    ctx->Zlast = Z;
    ctx->zscale = 1.0 / ss;
    }
    mark(ctx, s, e_ns);
    nv.next("mbd gradient");
    if (want_grad) {
        if (const int rg = backward_periodic(ctx, s, b, nullptr, out.grad_coords, out.grad_params)) return rg;
    }
    if (out.alpha_scs)
        MBD_CUDA(cudaMemcpyAsync(out.alpha_scs, ctx->dabar0, sizeof(double) * N, cudaMemcpyDeviceToDevice, s),
                 "outputs");
    mark(ctx, s, e_grad);
    MBD_CUDA(cudaStreamSynchronize(s), "mbd_evaluate");
    MBD_CUDA(cudaGetLastError(), "mbd_evaluate");
    ctx->prof.launches = static_cast<int>(launch_count() - launches0);
    if (ctx->profiling) {
        mbd_profile &p = ctx->prof;
        p.gemm_launches = (ctx->crt ? 1 : 4) * static_cast<int>(gemms.size());
        for (const Span &sp : gemms) {
            p.gemm_ms += span_ms(sp.a, sp.b);
            p.gemm_flops += sp.flops;
        }
        p.tc_launches = static_cast<int>(tc_spans.size());
        for (const Span &sp : tc_spans) {
            p.tc_ms += span_ms(sp.a, sp.b);
            p.tc_flops += sp.flops;
        }
        p.screening_ms = span_ms(e_start, e_scs);
        p.screening_flops = ctx->opt.scs_mode == MBD_SCS_NL ? 0.0 : nf1 * nd * nd * nd / 3.0;
        p.newton_schulz_ms = span_ms(e_scs, e_ns);
        p.gradient_ms = span_ms(e_ns, e_grad);
        p.total_ms = span_ms(e_start, e_grad);
    }
    ctx->have_result = true;
    ctx->have_forward = true;
    ++ctx->eval_count;
    return MBD_OK;
}

int run(mbd_ctx *ctx, cudaStream_t s, const Inputs &in, const Outputs &out, bool want_grad) {
    if (ctx->periodic) return run_periodic(ctx, s, in, out, want_grad);
    const int N = ctx->N, n = ctx->n, nf1 = ctx->nf1;
    const long long ld = ctx->ld, mat = ld * ld, xs = 3 * ld;
    const double beta = ctx->opt.beta, a = ctx->opt.a;
    ctx->have_result = false;
    ctx->have_screening = false;
    ctx->tq_valid = false;
    ctx->ev_used = 0;
    ctx->prof = mbd_profile{};
    const long long launches0 = launch_count();
    cudaEvent_t e_start = nullptr, e_scs = nullptr, e_ns = nullptr, e_grad = nullptr, e_corr = nullptr;
    std::vector<Span> gemms, tc_spans;
    auto timed_gemm = [&](const GemmArgs &g, double flops) {
        Span sp;
        sp.flops = flops;
        mark(ctx, s, sp.a);
        gemm_f64(g, s);
        mark(ctx, s, sp.b);
        if (ctx->profiling) gemms.push_back(sp);
    };
    const double nd = static_cast<double>(ctx->n);
    const double flops_full = 2.0 * nd * nd * nd, flops_sym = nd * nd * (nd + 1.0);
    ctx->have_forward = false;
    const AtomBufs b = atom_bufs(ctx, in);
    NvtxStages nv;
    nv.next("mbd screening");
    mark(ctx, s, e_start);
    MBD_CUDA(cudaMemsetAsync(ctx->dstatus, 0, sizeof(int), s), "mbd_evaluate");
    // ---- screening (Sec. 2.3) ----
    const bool learned = ctx->opt.scs_mode == MBD_SCS_LEARNED && !ctx->force_plain;
    ctx->last_learned = false;
    if (learned) {   // model prediction of alpha_bar(iu) in place of the Dyson solves
        if (out.grad_params)
            return fail(ctx, MBD_ERR_UNSUPPORTED, "learned_screening",
                        "learned screening gives energies and coordinate gradients only");
        if (ctx->members < 1) return fail(ctx, MBD_ERR_STATE, "learned_screening", "no model set");
        int rc0 = ensure_learned(ctx);
        if (rc0) return rc0;
        prepare_atoms(b, ctx->dstatus, s);
        scs_features(N, 1, ctx->doffs, in.R, in.a0ref, in.c6ref, in.rref, in.ratio, ctx->dfeat, ctx->dmoments, s);
        const cudaError_t ef = mlp_forward(N, ctx->members, ctx->dfeat, ctx->dmeanstd, ctx->dmeanstd + kLF, ctx->dmodel,
                                           ctx->dYl, want_grad ? ctx->dzc : nullptr, s, nullptr, ctx->dpacked);
        if (ef != cudaSuccess) return cuda_fail(ctx, "learned_screening", ef);
        learned_alpha(N, ctx->members, nf1, ctx->dalu, ctx->dYl, ctx->dabar, ctx->dspread, s);
        screened_params(b, ctx->dstatus, s);
    } else if (ctx->opt.scs_mode == MBD_SCS_NL) {   // MBD-NL: oscillators set directly, no screening
        nl_params(b, ctx->dstatus, s);
    } else {
        prepare_atoms(b, ctx->dstatus, s);
        build_scs(b, beta, a, ctx->dM, ld, mat, ctx->dstatus, s);
        if (fp64_path(ctx->opt.precision)) {
            if (const int rf = factorise(ctx, ctx->dM, nf1, s, "screening")) return rf;
            init_rhs_identity(ctx->dX, ld, n, nf1, xs, s);
            chol_solve3_f64(ctx->dM, ld, mat, nf1, ctx->ddinv, ctx->dX, ctx->dB, xs, s);
        } else {   // FP32 factors, FP64-refined solutions
            MBD_CUDA(cholesky_f32_from_f64(ctx->dM, ctx->sM, ld, nf1, ctx->sdinv, ctx->spanel, ctx->dstatus, s),
                     "screening");
            init_rhs_identity(ctx->dB, ld, n, nf1, xs, s);
            refine_solve3(ctx->dM, ctx->sM, ctx->sdinv, ld, n, nf1, ctx->dB, ctx->dX, ctx->swork, kRefineSteps, s);
        }
        contract_screen(b, ctx->dX, ld, xs, ctx->dstatus, s);
    }
    mark(ctx, s, e_scs);
    nv.next("mbd coupled oscillators and Newton-Schulz");
    int rc = read_status(ctx, s, "screening");
    if (rc) return rc;
    ctx->have_screening = true;
    // ---- coupled-oscillator matrix and its square roots (Sec. 2.1) ----
    build_q(b, beta, a, ctx->dQ, ld, ctx->dstatus, s);
    max_abs_rowsum(ctx->dQ, ld, static_cast<int>(ld), ctx->dscal + 1, s);
    double sc = 0.0;
    MBD_CUDA(cudaMemcpyAsync(&sc, ctx->dscal + 1, sizeof(double), cudaMemcpyDeviceToHost, s), "newton_schulz");
    MBD_CUDA(cudaStreamSynchronize(s), "newton_schulz");
    rc = read_status(ctx, s, "coupled_oscillator_matrix");
    if (rc) return rc;
    if (!(sc > 0.0) || !std::isfinite(sc)) return fail(ctx, MBD_ERR_INPUT, "newton_schulz", "invalid Q scale");
    // Lanczos estimates of the extreme eigenvalues of Q (workspace: rows of P).  The
    // largest tightens the scale s of Y0 = Q/s (Lanczos converges fast at the top of the
    // spectrum; a 5 % margin keeps Y0's spectrum inside (0, 1]).  The smallest converges
    // slowly: after 48 steps its Ritz value is 3-6 times the smallest eigenvalue of Q
    // (500-2000 atom clusters), so a quarter of it is the lower bound of the scaled
    // iteration.  A bound on either side of the true one only costs steps (see below); on the
    // spectra of those clusters a quarter takes one step fewer than a half.
    const bool short_run = !fp64_path(ctx->opt.precision) && ld <= kLanczosSmallOrder;
    const int lz_steps = std::min(short_run ? kLanczosStepsSmall : kLanczosSteps, static_cast<int>(ld));
    if (fp64_path(ctx->opt.precision))
        lanczos_coefficients(ctx->dQ, ld, lz_steps, ctx->dP, ctx->dscal + 8, s);
    else   // the bounds need a few digits; the products read an FP32 copy of Q (in the FP32 Y buffer)
        lanczos_coefficients_f32(ctx->dQ, ctx->fY, ld, lz_steps, ctx->dP, ctx->dscal + 8, s);
    std::vector<double> lz(2 * lz_steps);
    MBD_CUDA(cudaMemcpyAsync(lz.data(), ctx->dscal + 8, sizeof(double) * 2 * lz_steps, cudaMemcpyDeviceToHost, s),
             "newton_schulz");
    MBD_CUDA(cudaStreamSynchronize(s), "newton_schulz");
    double th_min = 0.0, th_max = sc;
    {
        std::vector<double> da, db;
        for (int j = 0; j < lz_steps; ++j) {
            da.push_back(lz[2 * j]);
            if (j + 1 < lz_steps) db.push_back(lz[2 * j + 1]);
            if (!(lz[2 * j + 1] > 1e-14 * sc)) break;   // invariant subspace reached
        }
        db.resize(da.size() > 0 ? da.size() - 1 : 0);
        if (!da.empty()) tridiag_extremes(da, db, th_min, th_max);
    }
    // ubound: upper bound on sqrt(eig(Z Y)) for the first step: 1 under the Gershgorin
    // scale; 1.05 after tightening by the Lanczos estimate (tolerates an underestimate
    // of the largest eigenvalue by up to 16 %).
    double ubound = 1.0;
    if (std::isfinite(th_max) && th_max > 0.0 && 1.05 * th_max < sc) {
        sc = 1.05 * th_max;
        ubound = 1.05;
    }
    ctx->ns_scale = sc;
    double lbound = ns::lower_estimate(th_min, sc);   // estimated lower bound on sqrt(eig(Z Y))
    const double ss = std::sqrt(sc);
    double *energy_out = out.energy ? out.energy : ctx->dscal;
    if (fp64_path(ctx->opt.precision)) {
        double *Y = ctx->dQ, *Z = ctx->dZ, *P = ctx->dP, *Y2 = ctx->dY2, *Z2 = ctx->dZ2;
        scale_matrix(Y, ld, 1.0 / sc, s);
        set_identity(Z, ld, s);
        const int M = static_cast<int>(ld);
        CrtProducts crt(ctx, s);
        cudaError_t ce = cudaSuccess;
        bool converged = false;
        double resid = 0.0;
        int it = 0;
        for (; it < ctx->opt.ns_max_iter; ++it) {
            // P = Z Y (not symmetric once rounding separates Z and Y; computed in full)
            const double *Pk = Y;   // Z_0 = I: P_0 = Y_0
            if (it > 0) {
                if (ctx->crt) {
                    Span sp;
                    sp.flops = flops_full;
                    mark(ctx, s, sp.a);
                    ce = crt.product(Z, Y, P, ctx->dPT);
                    mark(ctx, s, sp.b);
                    if (ctx->profiling) gemms.push_back(sp);
                    if (ce != cudaSuccess) return cuda_fail(ctx, "newton_schulz", ce);
                } else {
                    GemmArgs g{Z, Y, nullptr, P, ld, ld, 0, ld, 0, 0, 0, 0, M, M, M, 1, 1.0, 0.0, 0, 0};
                    timed_gemm(g, flops_full);
                }
                Pk = P;
            }
            frob_dev_identity(Pk, ld, n, ctx->dscal + 2, s);
            double r2 = 0.0;
            MBD_CUDA(cudaMemcpyAsync(&r2, ctx->dscal + 2, sizeof(double), cudaMemcpyDeviceToHost, s), "newton_schulz");
            MBD_CUDA(cudaStreamSynchronize(s), "newton_schulz");
            resid = std::sqrt(r2);
            if (!std::isfinite(resid) || resid > 2.0 * std::sqrt(static_cast<double>(n)) + 1.0) {
                // For positive definite Q every eigenvalue of Z Y stays in (0, 1]; leaving that
                // range means an eigenvalue of Q is not positive.
                ctx->ns_iter = it;
                ctx->ns_resid = resid;
                return fail(ctx, MBD_ERR_NEG_EIGENVALUE, "newton_schulz",
                            "Q has a non-positive eigenvalue (polarization catastrophe)");
            }
            const bool last = resid < ctx->opt.ns_tol;
            const ns::Coeffs cf = ns::step(lbound, ubound, last);   // scaled step (ns_schedule.h)
            const double c1 = cf.c1, c3 = cf.c3;
            // Y' = Y T, Z' = T Z: Y' = c1 Y + c3 Y (Z Y) and Z' = c1 Z + c3 (Z Y) Z.  Y Z Y and
            // Z Y Z are symmetric for any symmetric Y, Z, so only their upper tiles are
            // computed.  (Using P^T in place of P, i.e. Y Y Z, breaks the coupling and makes
            // rounding errors grow by about sqrt(cond Q)/2 per step.)
            if (ctx->crt) {
                Span sp;
                sp.flops = it == 0 ? flops_sym : 2.0 * flops_sym;
                mark(ctx, s, sp.a);
                ce = it == 0 ? crt.first_step(Y, Y2, c1, c3) : crt.step(Y, Z, P, ctx->dPT, Y2, Z2, c1, c3);
                mark(ctx, s, sp.b);
                if (ctx->profiling) gemms.push_back(sp);
                if (ce != cudaSuccess) return cuda_fail(ctx, "newton_schulz", ce);
            } else {
                GemmArgs gy{Y, Pk, Y, Y2, ld, ld, ld, ld, 0, 0, 0, 0, M, M, M, 1, c3, c1, 2, 0};
                timed_gemm(gy, flops_sym);
                if (it > 0) {
                    GemmArgs gz{Pk, Z, Z, Z2, ld, ld, ld, ld, 0, 0, 0, 0, M, M, M, 1, c3, c1, 2, 0};
                    timed_gemm(gz, flops_sym);
                }
            }
            if (it == 0) axpby_identity(Z2, Pk, ld, c1, c3, s);
            std::swap(Y, Y2);
            std::swap(Z, Z2);
            if (last) {
                converged = true;
                ++it;
                break;
            }
        }
        ctx->ns_iter = it;
        ctx->ns_resid = resid;
        if (ctx->crt) {   // tensor-core waits are bounded: check them
            int st = 0;
            MBD_CUDA(cudaMemcpyAsync(&st, ctx->dstatus, sizeof(int), cudaMemcpyDeviceToHost, s), "newton_schulz");
            MBD_CUDA(cudaStreamSynchronize(s), "newton_schulz");
            if (st & ST_TC_TIMEOUT) return fail(ctx, MBD_ERR_CUDA, "newton_schulz", "tensor-core GEMM wait timed out");
        }
        if (!converged)
            return fail(ctx, MBD_ERR_NOT_CONVERGED, "newton_schulz", "iteration cap reached");
        energy_trace(Y, ld, n, ctx->dombar, N, ss, energy_out, s);
        ctx->Zlast = Z;
        ctx->zscale = 1.0 / ss;
    } else {
        const MixProblem pr{ctx->dQ, ld, n, ctx->dP, ctx->dZ2, ctx->dY2, ctx->dZ, ctx->dtq, energy_out};
        std::vector<MixItem> items(1);
        items[0].sc = sc, items[0].lbound = lbound, items[0].ubound = ubound;
        rc = newton_schulz_mixed(ctx, s, pr, items, tc_spans, e_corr);
        if (rc) return rc;
        ctx->tq_valid = true;
    }
    mark(ctx, s, e_ns);
    nv.next("mbd gradient");
    if (learned) {
        // energy-error estimate from the adjoints h = dE/d alpha_bar(u) and the members' spread;
        // above the threshold the evaluation is redone with plain screening
        MbdGradOut go{ctx->dgomb, ctx->dgab0, ctx->dgrb, ctx->dgR};
        mbd_grad_pass(b, beta, a, ctx->Zlast, ld, ctx->zscale, go, s, ctx->tq_valid ? ctx->dtq : nullptr);
        chain_screen(b, go, ctx->dh, ctx->dga0, ctx->dgrv, ctx->dV, ld, xs, s);
        learned_estimate(N, nf1, ctx->members, ctx->opt.learned_estimate_scale, ctx->dh, ctx->dalu, ctx->dYl,
                         ctx->dscal + 5, s);
        double est = 0.0;
        MBD_CUDA(cudaMemcpyAsync(&est, ctx->dscal + 5, sizeof(double), cudaMemcpyDeviceToHost, s), "learned_screening");
        MBD_CUDA(cudaStreamSynchronize(s), "learned_screening");
        ctx->learned_est = est;
        ctx->learned_fallback = 0;
        ctx->last_learned = est <= ctx->opt.learned_max_error;
        if (!(est <= ctx->opt.learned_max_error)) {
            // the profile of the plain re-run also counts the discarded learned attempt
            const int attempt_launches = static_cast<int>(launch_count() - launches0);
            double attempt_ms = 0.0;
            if (ctx->profiling && e_start && e_ns) {
                MBD_CUDA(cudaEventSynchronize(e_ns), "learned_screening");
                attempt_ms = span_ms(e_start, e_ns);
            }
            ctx->force_plain = true;
            const int rc2 = run(ctx, s, in, out, want_grad);
            ctx->force_plain = false;
            ctx->learned_est = est;
            ctx->learned_fallback = 1;
            ctx->prof.launches += attempt_launches;
            ctx->prof.total_ms += attempt_ms;
            return rc2;
        }
        if (want_grad) {
            // dE/dR = (MBD term at fixed screened parameters, in dgR) + sum h dalpha_bar/dR through
            // the members' outputs, the network and the features
            learned_dy(N, ctx->members, nf1, ctx->dh, ctx->dabar, ctx->dYl, s);
            const cudaError_t eb = mlp_backward(N, ctx->members, ctx->dfeat, ctx->dmeanstd, ctx->dmeanstd + kLF,
                                                ctx->dmodel, ctx->dzc, ctx->dYl, ctx->dXl, nullptr, s, ctx->dpacked);
            if (eb != cudaSuccess) return cuda_fail(ctx, "learned_screening", eb);
            learned_forces(N, ctx->doffs, in.R, in.a0ref, in.rref, in.ratio, ctx->dmoments, ctx->dXl, ctx->members,
                           ctx->dadj, ctx->dgR, s);
            if (out.grad_coords) scale_copy(ctx->dgR, 3 * N, nullptr, out.grad_coords, s);
        }
    }
    // ---- gradients (Sec. 2.4) ----
    if (want_grad && !learned) backward_passes(ctx, s, b, nullptr, out.grad_coords, out.grad_params);
    if (out.alpha_scs)
        MBD_CUDA(cudaMemcpyAsync(out.alpha_scs, ctx->dabar0, sizeof(double) * N, cudaMemcpyDeviceToDevice, s),
                 "outputs");
    mark(ctx, s, e_grad);
    MBD_CUDA(cudaStreamSynchronize(s), "mbd_evaluate");
    MBD_CUDA(cudaGetLastError(), "mbd_evaluate");
    ctx->prof.launches = static_cast<int>(launch_count() - launches0);
    if (ctx->profiling) {
        mbd_profile &p = ctx->prof;
        p.gemm_launches = static_cast<int>(gemms.size());
        for (const Span &sp : gemms) {
            p.gemm_ms += span_ms(sp.a, sp.b);
            p.gemm_flops += sp.flops;
        }
        p.tc_launches = static_cast<int>(tc_spans.size());
        for (const Span &sp : tc_spans) {
            p.tc_ms += span_ms(sp.a, sp.b);
            p.tc_flops += sp.flops;
        }
        if (e_corr) p.correction_ms = span_ms(e_corr, e_ns);
        p.screening_ms = span_ms(e_start, e_scs);
        p.screening_flops = ctx->opt.scs_mode == MBD_SCS_NL
                                ? 0.0
                                : nf1 * nd * nd * nd / 3.0;   // FP64, or FP32 in the mixed modes
        p.newton_schulz_ms = span_ms(e_scs, e_ns);
        p.gradient_ms = span_ms(e_ns, e_grad);
        p.total_ms = span_ms(e_start, e_grad);
    }
    ctx->have_result = true;
    ctx->have_forward = true;
    ++ctx->eval_count;
    return MBD_OK;
}

}  // namespace

void mbdgb::set_scratch_limits(mbd_ctx *ctx, const ScratchLimits &lim) {
    ctx->lim = lim;
    release(ctx);   // the next mbd_set_geometry carves anew
    ctx->have_geom = ctx->have_params = ctx->have_forward = ctx->have_result = false;
}

extern "C" {

int mbd_default_options(mbd_options *opt) {
    if (!opt) return MBD_ERR_INPUT;
    opt->n_freq = 15;
    opt->beta = 0.83;
    opt->a = 6.0;
    opt->precision = MBD_PREC_FP64;
    opt->ns_tol = 1e-8;
    opt->ns_max_iter = 100;
    opt->tc_chunk_stages = 0;
    opt->ewald_gamma = 0.0;
    opt->real_cutoff = 0.0;
    opt->recip_cutoff = 0.0;
    opt->scs_mode = MBD_SCS_PLAIN;
    opt->learned_max_error = 1e-6;
    opt->mixed_max_error = 1e-7;
    opt->learned_estimate_scale = 1.0;
    return MBD_OK;
}

int mbd_create(mbd_ctx **out, int cuda_device, const mbd_options *opt) {
    if (!out) return MBD_ERR_INPUT;
    *out = nullptr;
    mbd_options o;
    if (opt) o = *opt; else mbd_default_options(&o);
    if (o.n_freq < 1 || o.n_freq + 1 > kMaxFreq || !(o.beta > 0) || !(o.a > 0) || o.ns_max_iter < 1 ||
        !(o.ns_tol > 0) || o.precision < MBD_PREC_FP64 || o.precision > MBD_PREC_FP64_SPLIT || o.tc_chunk_stages < 0 ||
        (o.scs_mode != MBD_SCS_PLAIN && o.scs_mode != MBD_SCS_LEARNED && o.scs_mode != MBD_SCS_NL) ||
        !(o.learned_max_error > 0) || !(o.mixed_max_error > 0) || !(o.learned_estimate_scale > 0) ||
        !std::isfinite(o.learned_estimate_scale) || (o.scs_mode == MBD_SCS_LEARNED && o.n_freq != 15))
        return MBD_ERR_INPUT;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || cuda_device < 0 || cuda_device >= ndev)
        return MBD_ERR_CUDA;
    mbd_ctx *c = new mbd_ctx();
    c->device = cuda_device;
    c->opt = o;
    c->nf1 = o.n_freq + 1;
    casimir_polder_grid(o.n_freq, c->hu, c->hwu);
    if (cudaSetDevice(cuda_device) != cudaSuccess ||
        cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking) != cudaSuccess) {
        delete c;
        return MBD_ERR_CUDA;
    }
    *out = c;
    return MBD_OK;
}

int mbd_destroy(mbd_ctx *ctx) {
    if (!ctx) return MBD_OK;
    cudaSetDevice(ctx->device);
    release(ctx);
    if (ctx->lslab) cudaFree(ctx->lslab);
    for (cudaEvent_t e : ctx->events) cudaEventDestroy(e);
    if (ctx->stream) cudaStreamDestroy(ctx->stream);
    scratch_trim(ctx->device);
    delete ctx;
    return MBD_OK;
}

int mbd_set_geometry(mbd_ctx *ctx, int n_atoms, const double *coords, const double *lattice,
                     const int *k_grid) {
    if (!ctx) return MBD_ERR_INPUT;
    if ((lattice == nullptr) != (k_grid == nullptr))
        return fail(ctx, MBD_ERR_INPUT, "mbd_set_geometry", "lattice and k_grid are given together or not at all");
    if (n_atoms < 1 || !coords) return fail(ctx, MBD_ERR_INPUT, "mbd_set_geometry", "need n_atoms >= 1 and coords");
    for (int k = 0; k < 3 * n_atoms; ++k)
        if (!std::isfinite(coords[k])) return fail(ctx, MBD_ERR_INPUT, "mbd_set_geometry", "non-finite coordinate");
    const bool periodic = lattice != nullptr;
    PeriodicSetup ps;
    if (periodic) {
        if (ctx->opt.precision == MBD_PREC_FP64_SPLIT)
            return fail(ctx, MBD_ERR_UNSUPPORTED, "mbd_set_geometry",
                        "periodic systems run in FP64 or in the tensor-core modes, not with split FP64 products");
        const int rc = periodic_setup(ctx->opt, lattice, k_grid, ps);
        if (rc) return fail(ctx, rc, "mbd_set_geometry", ps.msg);
    }
    MBD_CUDA(cudaSetDevice(ctx->device), "mbd_set_geometry");
    const bool realloc = (n_atoms != ctx->N) || !ctx->slab || periodic != ctx->periodic ||
                         (periodic && (ps.nk != ctx->nk || ps.nG != ctx->nG || ps.maxG != ctx->maxG));
    ctx->N = n_atoms;
    ctx->n = 3 * n_atoms;
    ctx->ld = (ctx->n + 127) / 128 * 128;   // 128: the tensor-core tile (also a multiple of 64)
    ctx->lde = (2LL * ctx->n + 127) / 128 * 128;
    ctx->nb = static_cast<int>(ctx->ld / kTile);
    ctx->hR.assign(coords, coords + 3 * n_atoms);
    ctx->periodic = periodic;
    if (periodic) {
        ctx->cell = ps.cell;
        ctx->nk = ps.nk;
        ctx->nkt = ps.nkt;
        ctx->hkw = ps.kw;
        ctx->nG = ps.nG;
        ctx->maxG = ps.maxG;
        ctx->hkq = ps.kq;
        ctx->hG = ps.G;
        ctx->hglist = ps.glist;
        ctx->hgcount = ps.gcount;
    } else {
        ctx->nk = ctx->nkt = 1;
        ctx->nG = ctx->maxG = 0;
    }
    ctx->have_lattice_grad = false;
    if (realloc) {
        ctx->have_params = false;
        ctx->have_forward = false;
        int rc = allocate(ctx);
        if (rc) { ctx->have_geom = false; return rc; }
    }
    if (periodic) {
        // The image tables' size depends on the lattice.  More scratch for a changed one comes beside the slab, whose
        // parameters and last evaluation stay; where it does not fit, the cell takes the direct kernels.
        const size_t need = ctx->no_scratch ? 0 : cell_products_bytes(n_atoms, ps.cell, ps.nk, ps.maxG, ctx->opt.precision, ctx->lim);
        void *more = nullptr;
        if (need > ctx->qwork_bytes) {
            if (cudaMalloc(&more, need) == cudaSuccess) {
                if (ctx->qslab) cudaFree(ctx->qslab);
                ctx->qslab = more;
                ctx->qwork = static_cast<char *>(more);
                ctx->qwork_bytes = need;
            } else {
                cudaGetLastError();
            }
        }
        const int rc = upload_periodic(ctx);
        if (rc) { ctx->have_geom = false; return rc; }
    }
    ctx->have_geom = true;
    ctx->have_result = false;
    return MBD_OK;
}

int mbd_set_free_atom_params(mbd_ctx *ctx, const double *alpha0_ref, const double *c6_ref,
                             const double *rvdw_ref, const double *volume_ratio) {
    if (!ctx) return MBD_ERR_INPUT;
    if (!ctx->have_geom) return fail(ctx, MBD_ERR_STATE, "mbd_set_free_atom_params", "set the geometry first");
    if (!alpha0_ref || !c6_ref || !rvdw_ref || !volume_ratio)
        return fail(ctx, MBD_ERR_INPUT, "mbd_set_free_atom_params", "null parameter array");
    const int N = ctx->N;
    ctx->ha0.assign(alpha0_ref, alpha0_ref + N);
    ctx->hc6.assign(c6_ref, c6_ref + N);
    ctx->hrr.assign(rvdw_ref, rvdw_ref + N);
    ctx->hv.assign(volume_ratio, volume_ratio + N);
    ctx->have_params = true;
    ctx->have_result = false;
    return MBD_OK;
}

int mbd_evaluate(mbd_ctx *ctx, double *energy, double *grad_coords, double *grad_lattice,
                 double *grad_params, double *alpha_scs) {
    if (!ctx) return MBD_ERR_INPUT;
    if (!ctx->have_geom || !ctx->have_params)
        return fail(ctx, MBD_ERR_STATE, "mbd_evaluate", "set the geometry and the free-atom parameters first");
    if (grad_lattice && !ctx->periodic)
        return fail(ctx, MBD_ERR_UNSUPPORTED, "mbd_evaluate", "no lattice gradient for finite systems");
    if (!energy) return fail(ctx, MBD_ERR_INPUT, "mbd_evaluate", "energy pointer is required");
    MBD_CUDA(cudaSetDevice(ctx->device), "mbd_evaluate");
    const int N = ctx->N;
    cudaStream_t s = ctx->stream;
    MBD_CUDA(cudaMemcpyAsync(ctx->dR, ctx->hR.data(), sizeof(double) * 3 * N, cudaMemcpyHostToDevice, s), "mbd_evaluate");
    MBD_CUDA(cudaMemcpyAsync(ctx->da0ref, ctx->ha0.data(), sizeof(double) * N, cudaMemcpyHostToDevice, s), "mbd_evaluate");
    MBD_CUDA(cudaMemcpyAsync(ctx->dc6ref, ctx->hc6.data(), sizeof(double) * N, cudaMemcpyHostToDevice, s), "mbd_evaluate");
    MBD_CUDA(cudaMemcpyAsync(ctx->drref, ctx->hrr.data(), sizeof(double) * N, cudaMemcpyHostToDevice, s), "mbd_evaluate");
    MBD_CUDA(cudaMemcpyAsync(ctx->dratio, ctx->hv.data(), sizeof(double) * N, cudaMemcpyHostToDevice, s), "mbd_evaluate");
    const bool want_grad = grad_coords || grad_params || grad_lattice;
    Inputs in{ctx->dR, ctx->da0ref, ctx->dc6ref, ctx->drref, ctx->dratio};
    Outputs o{ctx->dscal, nullptr, grad_params ? ctx->dgp : nullptr, nullptr};   // gradients stay in dgR
    int rc = run(ctx, s, in, o, want_grad);
    if (rc) return rc;
    double e = 0.0;
    MBD_CUDA(cudaMemcpyAsync(&e, ctx->dscal, sizeof(double), cudaMemcpyDeviceToHost, s), "mbd_evaluate");
    if (grad_coords)
        MBD_CUDA(cudaMemcpyAsync(grad_coords, ctx->dgR, sizeof(double) * 3 * N, cudaMemcpyDeviceToHost, s), "mbd_evaluate");
    if (grad_params)
        MBD_CUDA(cudaMemcpyAsync(grad_params, ctx->dgp, sizeof(double) * 4 * N, cudaMemcpyDeviceToHost, s), "mbd_evaluate");
    if (alpha_scs)
        MBD_CUDA(cudaMemcpyAsync(alpha_scs, ctx->dabar0, sizeof(double) * N, cudaMemcpyDeviceToHost, s), "mbd_evaluate");
    if (grad_lattice)
        MBD_CUDA(cudaMemcpyAsync(grad_lattice, ctx->dgAout, sizeof(double) * 9, cudaMemcpyDeviceToHost, s), "mbd_evaluate");
    MBD_CUDA(cudaStreamSynchronize(s), "mbd_evaluate");
    *energy = e;
    return MBD_OK;
}

int mbd_evaluate_dev(mbd_ctx *ctx, void *stream, int n_atoms, const double *coords, const double *alpha0_ref,
                     const double *c6_ref, const double *rvdw_ref, const double *volume_ratio, double *energy,
                     double *grad_coords, double *grad_params, double *alpha_scs) {
    if (!ctx) return MBD_ERR_INPUT;
    if (!ctx->have_geom) return fail(ctx, MBD_ERR_STATE, "mbd_evaluate_dev", "set the geometry first");
    if (n_atoms != ctx->N)
        return fail(ctx, MBD_ERR_INPUT, "mbd_evaluate_dev", "n_atoms differs from the geometry's size");
    if (!coords || !alpha0_ref || !c6_ref || !rvdw_ref || !volume_ratio || !energy)
        return fail(ctx, MBD_ERR_INPUT, "mbd_evaluate_dev", "null device pointer");
    MBD_CUDA(cudaSetDevice(ctx->device), "mbd_evaluate_dev");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const bool want_grad = grad_coords || grad_params;
    Inputs in{coords, alpha0_ref, c6_ref, rvdw_ref, volume_ratio};
    Outputs o{energy, grad_coords, grad_params, alpha_scs};
    return run(ctx, s, in, o, want_grad);
}

int mbd_get_evaluation_count(const mbd_ctx *ctx, long long *count) {
    if (!ctx || !count) return MBD_ERR_INPUT;
    *count = ctx->eval_count;
    return MBD_OK;
}

int mbd_backward_dev(mbd_ctx *ctx, void *stream, long long evaluation, int n_atoms, const double *coords,
                     const double *alpha0_ref, const double *c6_ref, const double *rvdw_ref,
                     const double *volume_ratio, const double *grad_energy, double *grad_coords,
                     double *grad_params) {
    if (!ctx) return MBD_ERR_INPUT;
    if (!ctx->have_forward)
        return fail(ctx, MBD_ERR_STATE, "mbd_backward_dev", "no forward evaluation to differentiate");
    if (evaluation != 0 && evaluation != ctx->eval_count)
        return fail(ctx, MBD_ERR_STATE, "mbd_backward_dev",
                    "the context's last evaluation is not the one to differentiate (evaluate it again first)");
    if (ctx->last_learned)
        return fail(ctx, MBD_ERR_UNSUPPORTED, "mbd_backward_dev",
                    "the last evaluation used learned screening; request its gradients from the evaluation");
    if (n_atoms != ctx->N || !coords || !alpha0_ref || !c6_ref || !rvdw_ref || !volume_ratio)
        return fail(ctx, MBD_ERR_INPUT, "mbd_backward_dev", "inputs must match the forward evaluation");
    MBD_CUDA(cudaSetDevice(ctx->device), "mbd_backward_dev");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    Inputs in{coords, alpha0_ref, c6_ref, rvdw_ref, volume_ratio};
    if (ctx->periodic) {
        if (const int rc = backward_periodic(ctx, s, atom_bufs(ctx, in), grad_energy, grad_coords, grad_params)) return rc;
    } else backward_passes(ctx, s, atom_bufs(ctx, in), grad_energy, grad_coords, grad_params);
    MBD_CUDA(cudaStreamSynchronize(s), "mbd_backward_dev");
    MBD_CUDA(cudaGetLastError(), "mbd_backward_dev");
    return MBD_OK;
}

int mbd_set_scs_model(mbd_ctx *ctx, int n_members, const void *params_fp16, const float *mean, const float *std) {
    if (!ctx) return MBD_ERR_INPUT;
    if (n_members < 1 || n_members > 64 || !params_fp16 || !mean || !std)
        return fail(ctx, MBD_ERR_INPUT, "mbd_set_scs_model", "need 1..64 members, parameters, mean and std");
    for (int k = 0; k < kLF; ++k)
        if (!(std[k] > 0.0f) || !std::isfinite(mean[k]))
            return fail(ctx, MBD_ERR_INPUT, "mbd_set_scs_model", "feature std must be positive and mean finite");
    const size_t P = static_cast<size_t>(learned_param_count()) * n_members;
    const uint16_t *src = static_cast<const uint16_t *>(params_fp16);
    ctx->hmodel.assign(src, src + P);
    ctx->hmean.assign(mean, mean + kLF);
    ctx->hstd.assign(std, std + kLF);
    ctx->members = n_members;
    ctx->model_dirty = true;
    return MBD_OK;
}

int mbd_get_learned_stats(mbd_ctx *ctx, double *estimated_error, int *fell_back) {
    if (!ctx) return MBD_ERR_INPUT;
    if (estimated_error) *estimated_error = ctx->learned_est;
    if (fell_back) *fell_back = ctx->learned_fallback;
    return MBD_OK;
}

int mbd_screen(mbd_ctx *ctx, double *alpha_iu, double *alpha_free_iu, double *c6, double *omega, double *rvdw) {
    if (!ctx) return MBD_ERR_INPUT;
    if (!ctx->have_geom || !ctx->have_params)
        return fail(ctx, MBD_ERR_STATE, "mbd_screen", "set the geometry and the free-atom parameters first");
    if (ctx->opt.scs_mode == MBD_SCS_NL)
        return fail(ctx, MBD_ERR_UNSUPPORTED, "mbd_screen", "MBD-NL has no screening step");
    MBD_CUDA(cudaSetDevice(ctx->device), "mbd_screen");
    const int N = ctx->N, n = ctx->n, nf1 = ctx->nf1;
    const long long ld = ctx->ld, mat = ld * ld, xs = 3 * ld;
    cudaStream_t s = ctx->stream;
    MBD_CUDA(cudaMemcpyAsync(ctx->dR, ctx->hR.data(), sizeof(double) * 3 * N, cudaMemcpyHostToDevice, s), "mbd_screen");
    MBD_CUDA(cudaMemcpyAsync(ctx->da0ref, ctx->ha0.data(), sizeof(double) * N, cudaMemcpyHostToDevice, s), "mbd_screen");
    MBD_CUDA(cudaMemcpyAsync(ctx->dc6ref, ctx->hc6.data(), sizeof(double) * N, cudaMemcpyHostToDevice, s), "mbd_screen");
    MBD_CUDA(cudaMemcpyAsync(ctx->drref, ctx->hrr.data(), sizeof(double) * N, cudaMemcpyHostToDevice, s), "mbd_screen");
    MBD_CUDA(cudaMemcpyAsync(ctx->dratio, ctx->hv.data(), sizeof(double) * N, cudaMemcpyHostToDevice, s), "mbd_screen");
    const AtomBufs b = atom_bufs(ctx, Inputs{ctx->dR, ctx->da0ref, ctx->dc6ref, ctx->drref, ctx->dratio});
    ctx->have_screening = false;
    MBD_CUDA(cudaMemsetAsync(ctx->dstatus, 0, sizeof(int), s), "mbd_screen");
    prepare_atoms(b, ctx->dstatus, s);
    if (ctx->periodic) build_scs_periodic(b, ctx->cell, ctx->opt.beta, ctx->opt.a, ctx->dM, ld, mat, ctx->dstatus, s);
    else build_scs(b, ctx->opt.beta, ctx->opt.a, ctx->dM, ld, mat, ctx->dstatus, s);
    if (fp64_path(ctx->opt.precision) || ctx->periodic) {
        if (const int rf = factorise(ctx, ctx->dM, nf1, s, "mbd_screen")) return rf;
        init_rhs_identity(ctx->dX, ld, n, nf1, xs, s);
        chol_solve3_f64(ctx->dM, ld, mat, nf1, ctx->ddinv, ctx->dX, ctx->dB, xs, s);
    } else {
        MBD_CUDA(cholesky_f32_from_f64(ctx->dM, ctx->sM, ld, nf1, ctx->sdinv, ctx->spanel, ctx->dstatus, s),
                 "mbd_screen");
        init_rhs_identity(ctx->dB, ld, n, nf1, xs, s);
        refine_solve3(ctx->dM, ctx->sM, ctx->sdinv, ld, n, nf1, ctx->dB, ctx->dX, ctx->swork, kRefineSteps, s);
    }
    contract_screen(b, ctx->dX, ld, xs, ctx->dstatus, s);
    int rc = read_status(ctx, s, "mbd_screen");
    if (rc) return rc;
    ctx->have_screening = true;
    if (alpha_free_iu)
        MBD_CUDA(cudaMemcpy(alpha_free_iu, ctx->dalu, sizeof(double) * N * nf1, cudaMemcpyDeviceToHost), "mbd_screen");
    return mbd_get_scs_detail(ctx, alpha_iu, c6, omega, rvdw);
}

int mbd_get_lattice_gradient(mbd_ctx *ctx, double *grad_lattice) {
    if (!ctx || !grad_lattice) return MBD_ERR_INPUT;
    if (!ctx->periodic || !ctx->have_lattice_grad)
        return fail(ctx, MBD_ERR_STATE, "mbd_get_lattice_gradient", "no lattice gradient has been computed");
    MBD_CUDA(cudaSetDevice(ctx->device), "mbd_get_lattice_gradient");
    MBD_CUDA(cudaMemcpy(grad_lattice, ctx->dgAout, sizeof(double) * 9, cudaMemcpyDeviceToHost), "mbd_get_lattice_gradient");
    return MBD_OK;
}

int mbd_get_scs_detail(mbd_ctx *ctx, double *alpha_iu, double *c6, double *omega, double *rvdw) {
    if (!ctx) return MBD_ERR_INPUT;
    if (!ctx->have_screening) return fail(ctx, MBD_ERR_STATE, "mbd_get_scs_detail", "no screening result");
    MBD_CUDA(cudaSetDevice(ctx->device), "mbd_get_scs_detail");
    const size_t N = ctx->N;
    if (alpha_iu) MBD_CUDA(cudaMemcpy(alpha_iu, ctx->dabar, sizeof(double) * N * ctx->nf1, cudaMemcpyDeviceToHost), "mbd_get_scs_detail");
    if (c6) MBD_CUDA(cudaMemcpy(c6, ctx->dc6bar, sizeof(double) * N, cudaMemcpyDeviceToHost), "mbd_get_scs_detail");
    if (omega) MBD_CUDA(cudaMemcpy(omega, ctx->dombar, sizeof(double) * N, cudaMemcpyDeviceToHost), "mbd_get_scs_detail");
    if (rvdw) MBD_CUDA(cudaMemcpy(rvdw, ctx->drbar, sizeof(double) * N, cudaMemcpyDeviceToHost), "mbd_get_scs_detail");
    return MBD_OK;
}

int mbd_ts_energy(mbd_ctx *ctx, double s_r, double *energy, double *grad_coords, double *grad_lattice,
                  double *grad_params) {
    if (!ctx) return MBD_ERR_INPUT;
    if (!energy || !(s_r > 0.0)) return fail(ctx, MBD_ERR_INPUT, "mbd_ts_energy", "energy is required; s_r > 0");
    if (!ctx->have_geom || !ctx->have_params)
        return fail(ctx, MBD_ERR_STATE, "mbd_ts_energy", "set the geometry and the free-atom parameters first");
    if (grad_lattice && !ctx->periodic)
        return fail(ctx, MBD_ERR_UNSUPPORTED, "mbd_ts_energy", "no lattice gradient for finite systems");
    if (ctx->opt.scs_mode == MBD_SCS_NL)
        return fail(ctx, MBD_ERR_UNSUPPORTED, "mbd_ts_energy", "TS takes the free-atom parameters of Eq. ts-scaling");
    MBD_CUDA(cudaSetDevice(ctx->device), "mbd_ts_energy");
    const int N = ctx->N;
    cudaStream_t s = ctx->stream;
    MBD_CUDA(cudaMemcpyAsync(ctx->dR, ctx->hR.data(), sizeof(double) * 3 * N, cudaMemcpyHostToDevice, s), "mbd_ts_energy");
    MBD_CUDA(cudaMemcpyAsync(ctx->da0ref, ctx->ha0.data(), sizeof(double) * N, cudaMemcpyHostToDevice, s), "mbd_ts_energy");
    MBD_CUDA(cudaMemcpyAsync(ctx->dc6ref, ctx->hc6.data(), sizeof(double) * N, cudaMemcpyHostToDevice, s), "mbd_ts_energy");
    MBD_CUDA(cudaMemcpyAsync(ctx->drref, ctx->hrr.data(), sizeof(double) * N, cudaMemcpyHostToDevice, s), "mbd_ts_energy");
    MBD_CUDA(cudaMemcpyAsync(ctx->dratio, ctx->hv.data(), sizeof(double) * N, cudaMemcpyHostToDevice, s), "mbd_ts_energy");
    MBD_CUDA(cudaMemsetAsync(ctx->dstatus, 0, sizeof(int), s), "mbd_ts_energy");
    const AtomBufs b = atom_bufs(ctx, Inputs{ctx->dR, ctx->da0ref, ctx->dc6ref, ctx->drref, ctx->dratio});
    prepare_atoms(b, ctx->dstatus, s);   // TS-scaled oscillators (Eq. ts-scaling) and input checks
    // scratch: partial sums in dM, per-atom energies in dh, dE/d(a0, om, rv) in dga0, dgom, dgrv (and for a cell
    // the lattice parts in dgApart, their sum in dgA); the next evaluation rewrites all of
    // them before use
    if (ctx->periodic) {
        const PeriodicBufs pb = periodic_bufs(ctx);
        structure_factors(b, pb, s);   // e^{i G.R_i} of the current coordinates
        ts_periodic(b, pb, s_r, ctx->dtsg, ctx->dh, ctx->dgR, ctx->dga0, ctx->dgom, ctx->dgrv, ctx->dgApart,
                    ctx->dgA, ctx->dstatus, s);
    } else {
        ts_pairs(b, s_r, ctx->dh, ctx->dgR, ctx->dga0, ctx->dgom, ctx->dgrv, ctx->dM, s);   // (dM: 144 N^2 doubles)
    }
    if (grad_params) ts_chain(b, ctx->dga0, ctx->dgom, ctx->dgrv, nullptr, ctx->dgp, s);
    std::vector<double> ea(N);
    MBD_CUDA(cudaMemcpyAsync(ea.data(), ctx->dh, sizeof(double) * N, cudaMemcpyDeviceToHost, s), "mbd_ts_energy");
    if (grad_coords)
        MBD_CUDA(cudaMemcpyAsync(grad_coords, ctx->dgR, sizeof(double) * 3 * N, cudaMemcpyDeviceToHost, s), "mbd_ts_energy");
    if (grad_lattice)
        MBD_CUDA(cudaMemcpyAsync(grad_lattice, ctx->dgA, sizeof(double) * 9, cudaMemcpyDeviceToHost, s), "mbd_ts_energy");
    if (grad_params)
        MBD_CUDA(cudaMemcpyAsync(grad_params, ctx->dgp, sizeof(double) * 4 * N, cudaMemcpyDeviceToHost, s), "mbd_ts_energy");
    ctx->have_forward = false;   // the gradient scratch of the last evaluation was reused
    int rc = read_status(ctx, s, "mbd_ts_energy");
    if (rc) return rc;
    double sum = 0.0, comp = 0.0;   // Neumaier sum of the per-atom energies
    for (double x : ea) {
        const double t = sum + x;
        comp += std::fabs(sum) >= std::fabs(x) ? (sum - t) + x : (x - t) + sum;
        sum = t;
    }
    *energy = sum + comp;
    return MBD_OK;
}

int mbd_log_energy(mbd_ctx *ctx, int max_order, double *energy, double *orders) {
    if (!ctx) return MBD_ERR_INPUT;
    if (!energy || max_order < 1 || max_order > 4 || (max_order > 1 && !orders))
        return fail(ctx, MBD_ERR_INPUT, "mbd_log_energy", "energy is required; max_order 1..4; orders for max_order > 1");
    if (ctx->periodic) return fail(ctx, MBD_ERR_UNSUPPORTED, "mbd_log_energy", "finite systems only");
    if (!ctx->have_screening)
        return fail(ctx, MBD_ERR_STATE, "mbd_log_energy", "no oscillators: evaluate the system first");
    MBD_CUDA(cudaSetDevice(ctx->device), "mbd_log_energy");
    cudaStream_t s = ctx->stream;
    const int N = ctx->N, nf = ctx->nf1 - 1;
    const long long ld = ctx->ld, mat = ld * ld;
    MBD_CUDA(cudaMemcpyAsync(ctx->dR, ctx->hR.data(), sizeof(double) * 3 * N, cudaMemcpyHostToDevice, s),
             "mbd_log_energy");
    MBD_CUDA(cudaMemsetAsync(ctx->dstatus, 0, sizeof(int), s), "mbd_log_energy");
    const AtomBufs b = atom_bufs(ctx, Inputs{ctx->dR, ctx->da0ref, ctx->dc6ref, ctx->drref, ctx->dratio});
    double *A = ctx->dM + mat;   // the nodes u_1..u_nf in screening slots 1..nf
    double *sums = ctx->dlog;    // [4][nf]: sum ln L_pp, Tr A^2, Tr A^3, Tr A^4
    MBD_CUDA(build_lr_freq(b, ctx->opt.beta, ctx->opt.a, A, ld, mat, nf, ctx->dstatus, s), "mbd_log_energy");
    if (max_order >= 2) MBD_CUDA(batch_dot(A, A, mat, mat, nf, sums + nf, s), "mbd_log_energy");   // A symmetric
    if (max_order >= 3) {
        const int M = static_cast<int>(ld);
        for (int k = 0; k < nf; ++k) {   // P = A_k^2 (symmetric), then <P, A_k> and |P|^2
            GemmArgs g{A + k * mat, A + k * mat, nullptr, ctx->dP, ld, ld, 0, ld, 0, 0, 0, 0, M, M, M, 1, 1.0, 0.0, 2, 0};
            gemm_f64(g, s);
            MBD_CUDA(batch_dot(ctx->dP, A + k * mat, mat, 0, 1, sums + 2 * nf + k, s), "mbd_log_energy");
            if (max_order >= 4) MBD_CUDA(batch_dot(ctx->dP, ctx->dP, mat, 0, 1, sums + 3 * nf + k, s), "mbd_log_energy");
        }
    }
    add_identity_batch(A, ld, mat, nf, s);
    if (const int rf = factorise(ctx, A, nf, s, "mbd_log_energy")) return rf;
    logdiag_batch(A, ld, mat, nf, sums, ctx->dstatus, s);
    std::vector<double> h(4 * nf);
    MBD_CUDA(cudaMemcpyAsync(h.data(), sums, sizeof(double) * 4 * nf, cudaMemcpyDeviceToHost, s), "mbd_log_energy");
    ctx->have_forward = false;   // the screening buffers now hold these factors
    int rc = read_status(ctx, s, "mbd_log_energy");
    if (rc) return rc;
    const double inv2pi = 1.0 / (2.0 * 3.141592653589793238462643383279502884);
    double e = 0.0;
    for (int k = 0; k < nf; ++k) e += ctx->hwu[k + 1] * 2.0 * h[k];   // ln det = 2 sum ln L_pp
    *energy = e * inv2pi;
    for (int m = 2; m <= max_order; ++m) {
        double t = 0.0;
        for (int k = 0; k < nf; ++k) t += ctx->hwu[k + 1] * h[(m - 1) * nf + k];
        orders[m - 2] = -inv2pi * ((m % 2 == 0) ? 1.0 : -1.0) / m * t;   // -(-1)^m/m Tr A^m
    }
    return MBD_OK;
}

int mbd_get_stats(mbd_ctx *ctx, int *ns_iterations, double *ns_scale, double *ns_residual,
                  double *correction_residual) {
    if (!ctx) return MBD_ERR_INPUT;
    if (correction_residual) *correction_residual = fp64_path(ctx->opt.precision) ? 0.0 : ctx->corr_resid;
    if (ns_iterations) *ns_iterations = ctx->ns_iter;
    if (ns_scale) *ns_scale = ctx->ns_scale;
    if (ns_residual) *ns_residual = ctx->ns_resid;
    return MBD_OK;
}

int mbd_get_workspace(const mbd_ctx *ctx, int *tensor_products, int *matrices_together) {
    if (!ctx) return MBD_ERR_INPUT;
    if (!ctx->have_geom) return MBD_ERR_STATE;
    if (tensor_products) *tensor_products = ctx->no_scratch ? 0 : 1;
    if (matrices_together) *matrices_together = ctx->mgroup;
    return MBD_OK;
}

int mbd_set_profiling(mbd_ctx *ctx, int enable) {
    if (!ctx) return MBD_ERR_INPUT;
    ctx->profiling = enable != 0;
    return MBD_OK;
}

int mbd_get_profile(mbd_ctx *ctx, mbd_profile *out) {
    if (!ctx || !out) return MBD_ERR_INPUT;
    *out = ctx->prof;
    return MBD_OK;
}

int mbd_get_exception(const mbd_ctx *ctx, int *code, char *origin, char *msg, size_t len) {
    if (!ctx) return MBD_ERR_INPUT;
    if (code) *code = ctx->err_code;
    if (origin && len) {
        std::strncpy(origin, ctx->err_origin.c_str(), len - 1);
        origin[len - 1] = '\0';
    }
    if (msg && len) {
        std::strncpy(msg, ctx->err_msg.c_str(), len - 1);
        msg[len - 1] = '\0';
    }
    return MBD_OK;
}

int mbdk_gemm_f64(void *stream, int trans_b, int mode, int M, int N, int K, double alpha,
                  const double *A, long long lda, const double *B, long long ldb, double beta,
                  const double *D, long long ldd, double *C, long long ldc) {
    if (M <= 0 || N <= 0 || K <= 0 || M % kTile || N % kTile || K % kTile || mode < 0 || mode > 3 ||
        (mode && M != N) || !A || !B || !C || (beta != 0.0 && !D) || (lda | ldb | ldc) & 1 ||
        (D && (ldd & 1)) || (trans_b != 0 && trans_b != 1))
        return MBD_ERR_INPUT;
    GemmArgs g{A, B, D, C, lda, ldb, ldd, ldc, 0, 0, 0, 0, M, N, K, 1, alpha, beta, mode, trans_b};
    gemm_f64(g, static_cast<cudaStream_t>(stream));
    return cudaGetLastError() == cudaSuccess ? MBD_OK : MBD_ERR_CUDA;
}

int mbdk_gemm_tc(void *stream, int kind, int mode, int M, int N, int K, float alpha, const void *A0,
                 const void *A1, long long lda, const void *B0, const void *B1, long long ldb, float beta,
                 const float *D, float *C, void *C_hi, void *C_lo, float *CT, long long ldc, int chunk_stages,
                 int *err) {
    if (!A0 || !B0 || (kind != 0 && (!A1 || !B1)) || ((C_hi != nullptr) != (C_lo != nullptr)) || chunk_stages < 0)
        return MBD_ERR_INPUT;
    TcOperands op{A0, kind != 0 ? A1 : A0, B0, kind != 0 ? B1 : B0, lda, ldb};
    TcArgs g{M, N, K, alpha, beta, D, ldc, C, C_hi, C_lo, CT, nullptr, nullptr, nullptr, 0, mode, err, nullptr,
             chunk_stages};
    const cudaError_t e = tc_gemm(kind, op, g, static_cast<cudaStream_t>(stream));
    if (e == cudaErrorInvalidValue) return MBD_ERR_INPUT;
    return e == cudaSuccess ? MBD_OK : MBD_ERR_CUDA;
}

int mbdk_tc_wait_check(void *stream, long long spin_cycles, int *err) {
    const cudaError_t e = tc_wait_probe(spin_cycles, err, static_cast<cudaStream_t>(stream));
    if (e == cudaErrorInvalidValue) return MBD_ERR_INPUT;
    return e == cudaSuccess ? MBD_OK : MBD_ERR_CUDA;
}

size_t mbdk_gemm_f64_split_work_bytes(int M, int N, int K) {
    if (M <= 0 || N <= 0 || K <= 0) return 0;
    return gemm_f64_split_work_bytes(M, N, K);
}

int mbdk_gemm_f64_split(void *stream, int trans_b, int M, int N, int K, double alpha, const double *A,
                        long long lda, const double *B, long long ldb, double beta, const double *D, long long ldd,
                        double *C, long long ldc, void *work, int *err) {
    if (M <= 0 || N <= 0 || K <= 0 || M % 128 || N % 128 || K % 64 || !A || !B || !C || !work || !err ||
        (beta != 0.0 && !D) || ldc % 8 || lda < K || ldb < (trans_b ? K : N) || ldc < N ||
        (D && D != C && ldd < N) || (trans_b != 0 && trans_b != 1))
        return MBD_ERR_INPUT;
    const cudaError_t e = gemm_f64_split(trans_b, 0, M, N, K, alpha, A, lda, B, ldb, beta, D, ldd, C, ldc, work, err,
                                         static_cast<cudaStream_t>(stream));
    if (e == cudaErrorInvalidValue) return MBD_ERR_INPUT;
    return e == cudaSuccess ? MBD_OK : MBD_ERR_CUDA;
}

int mbdk_cholesky_f64(void *stream, double *A, long long ld, int batch, double *dinv, int *status) {
    if (ld <= 0 || ld % kTile || batch < 1 || !A || !dinv || !status) return MBD_ERR_INPUT;
    cholesky_f64(A, ld, ld * ld, batch, dinv, status, static_cast<cudaStream_t>(stream));
    return cudaGetLastError() == cudaSuccess ? MBD_OK : MBD_ERR_CUDA;
}

int mbdk_chol_solve3_f64(void *stream, const double *L, long long ld, int batch, const double *dinv,
                         double *X, double *work) {
    if (ld <= 0 || ld % kTile || batch < 1 || !L || !dinv || !X || !work || work == X) return MBD_ERR_INPUT;
    chol_solve3_f64(L, ld, ld * ld, batch, dinv, X, work, 3 * ld, static_cast<cudaStream_t>(stream));
    return cudaGetLastError() == cudaSuccess ? MBD_OK : MBD_ERR_CUDA;
}

}  // extern "C"
