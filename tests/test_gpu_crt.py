"""FP64 products on the tensor cores by residues (csrc/k_crt.cu) at the edges of their tiles, stages,
accumulations and panels, against exact integers.

The bound is the arithmetic's own: each scaled row has a 2-norm of at least 0.65 2^58 and its
entries are rounded by at most 1/2, so a.b errs by at most 1.6 sqrt(K) 2^-58 |a| |b|; the way back
rounds to 64 bits of P (below 2^-60 |a| |b|) and to FP64 three times."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2308_03140_gb300 import binding, build

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def dev():
    build.build()
    binding.load()
    out = os.path.join(HERE, "_build")
    os.makedirs(out, exist_ok=True)
    so = os.path.join(out, "crt_device.so")
    libdir = os.path.dirname(build.LIB)
    cmd = [build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", f"-I{build.CSRC}",
           os.path.join(HERE, "crt_device.cu"), "-o", so, f"-L{libdir}", f"-l:{os.path.basename(build.LIB)}",
           "-Xlinker", f"-rpath={libdir}"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    L = C.CDLL(so)
    vp, i, ll, d = C.c_void_p, C.c_int, C.c_longlong, C.c_double
    L.crt_real_bytes.restype = L.crt_complex_bytes.restype = C.c_size_t
    L.crt_real.argtypes = [vp, ll, vp, ll, i, i, i, d, d, vp, ll, vp, ll, vp, ll, i, vp, vp]
    L.crt_complex.argtypes = [vp, vp, i, i, ll, i, d, d, vp, vp, vp, i, vp, vp]
    return L


def _cuda(x):
    import torch
    return torch.tensor(x, dtype=torch.float64, device="cuda:0")


def _p(t):
    return None if t is None else C.c_void_p(t.data_ptr())


def _even(x):
    return x + (x & 1)


def _padded(a, ld):
    out = np.full(a.shape[:-1] + (ld,), np.nan)    # what lies between the rows must not be read
    out[..., :a.shape[-1]] = a
    return _cuda(out)


def _call(L, A, B, alpha=1.0, beta=0.0, D=None, sym=False, transpose=False, alias=False):
    import torch
    M, K = A.shape
    N = B.shape[0]
    ld = _even(K)
    a, b = _padded(A, ld), _padded(B, ld)
    ldc = _even(N) + 2
    c = torch.full((M, ldc), 7.0, dtype=torch.float64, device="cuda:0")
    d = None if D is None else _padded(D, ldc)
    if alias:
        c = d
    t = torch.full((N, _even(M)), 7.0, dtype=torch.float64, device="cuda:0") if transpose else None
    work = torch.empty(int(L.crt_real_bytes(M, N, K)), dtype=torch.uint8, device="cuda:0")
    err = torch.zeros(1, dtype=torch.int32, device="cuda:0")
    rc = L.crt_real(_p(a), ld, _p(b), ld, M, N, K, alpha, beta, _p(d), ldc, _p(c), ldc, _p(t), _even(M), int(sym),
                    _p(work), _p(err))
    torch.cuda.synchronize()
    assert rc == 0 and int(err.item()) == 0
    return c.cpu().numpy()[:, :N], None if t is None else t.cpu().numpy()[:, :M]


def _ints(rng, rows, K, bits=24):
    """Integer rows of very different size (powers of two taken out: exact in FP64 and in int64)."""
    x = rng.integers(-2 ** bits, 2 ** bits, (rows, K))
    x[rng.random((rows, K)) < 0.3] //= 2 ** 12
    return x, rng.integers(-30, 30, rows)


def _check(got, exact, na, nb, K, alpha=1.0, extra=0.0):
    tol = abs(alpha) * 1.6 * np.sqrt(K) * 2.0 ** -58 * np.outer(na, nb) + 2.0 ** -51 * (np.abs(alpha * exact) + np.abs(extra))
    err = np.abs(got - (alpha * exact + extra))
    assert np.all(err <= tol), (err / tol).max()


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (3, 5, 7), (96, 96, 96), (128, 129, 64), (127, 255, 65), (256, 257, 512),
                                   (300, 130, 513), (257, 511, 1030), (40, 70, 2309)])
def test_real_products(dev, M, N, K):
    rng = np.random.default_rng(M + 7 * N + 31 * K)
    (xa, ea), (xb, eb) = _ints(rng, M, K), _ints(rng, N, K)
    exact = (xa @ xb.T).astype(np.float64) * np.ldexp(1.0, ea)[:, None] * np.ldexp(1.0, eb)[None, :]
    A, B = np.ldexp(xa.astype(np.float64), ea[:, None]), np.ldexp(xb.astype(np.float64), eb[:, None])
    na, nb = np.linalg.norm(A, axis=1), np.linalg.norm(B, axis=1)
    got, T = _call(dev, A, B, transpose=True)
    _check(got, exact, na, nb, K)
    assert np.array_equal(T, got.T)
    D = rng.normal(size=(M, N)) * np.outer(na, nb)
    got, _ = _call(dev, A, B, alpha=-0.5, beta=1.5, D=D, alias=True)
    _check(got, exact, na, nb, K, -0.5, 1.5 * D)


@pytest.mark.parametrize("n,K", [(3, 3), (96, 130), (257, 96), (513, 64)])
def test_symmetric_products(dev, n, K):
    # A A^T keeps its upper half, mirrored; D's lower half is not read
    rng = np.random.default_rng(n)
    x, _ = _ints(rng, n, K)
    A = x.astype(np.float64)
    D = rng.normal(size=(n, n)) * 2.0 ** 40
    D = D + D.T
    na = np.linalg.norm(A, axis=1)
    Du = np.where(np.tri(n, k=-1, dtype=bool), np.nan, D)
    got, _ = _call(dev, A, A, alpha=2.0, beta=-1.0, D=Du, sym=True, alias=True)
    _check(got, (x @ x.T).astype(np.float64), na, na, K, 2.0, -D)
    assert np.array_equal(got, got.T)


@pytest.mark.parametrize("K", [511, 512, 1024, 3000])
def test_largest_partial_sums(dev, K):
    # constant rows: every residue of a row is the same, so all products of an accumulation have one
    # sign and, for some moduli and rows, nearly the largest size
    rng = np.random.default_rng(K)
    a, b = rng.integers(2 ** 23, 2 ** 24, 200), rng.integers(2 ** 23, 2 ** 24, 180)
    A, B = np.repeat(a[:, None], K, 1).astype(np.float64), np.repeat(b[:, None], K, 1).astype(np.float64)
    got, _ = _call(dev, A, B)
    _check(got, np.outer(a, b).astype(np.float64) * K, a * np.sqrt(K), b * np.sqrt(K), K)


def test_zero_tiny_huge_and_bad_rows(dev):
    rng = np.random.default_rng(5)
    A, B = rng.normal(size=(7, 50)), rng.normal(size=(6, 50))
    A[1] = 0.0
    A[2] *= 1e-300
    A[3] *= 1e300
    A[4, 9] = np.nan
    B[2, 3] = np.inf
    B[4] *= 1e-290
    got, _ = _call(dev, A, B)
    assert np.all(np.isnan(got[4])) and np.all(np.isnan(got[:, 2]))
    ok = np.ix_([0, 1, 2, 3, 5, 6], [0, 1, 3, 4, 5])
    exact = A[ok[0].ravel()] @ B[ok[1].ravel()].T
    scale = np.outer(np.abs(A[ok[0].ravel()]).max(1), np.abs(B[ok[1].ravel()]).max(1))
    assert np.all(np.abs(got[ok] - exact) <= 1e-13 * scale + 1e-322)
    assert np.all(got[1, [0, 1, 3, 4, 5]] == 0.0)


def test_panels_of_long_rows(dev):
    rng = np.random.default_rng(6)
    n = 8300
    x = rng.integers(-2 ** 22, 2 ** 22, (n, n))
    A = x.astype(np.float64)
    na = np.linalg.norm(A, axis=1)
    rows = np.array([0, 1, 255, 8191, 8192, 8299])
    exact = (x[rows] @ x.T).astype(np.float64)
    got, T = _call(dev, A[:300], A, transpose=True)
    _check(got[rows[:3]], exact[:3], na[rows[:3]], na, n)
    assert np.array_equal(T, got.T)
    got, _ = _call(dev, A, A, sym=True)
    _check(got[rows], exact, na[rows], na, n)
    assert np.array_equal(got, got.T)


@pytest.mark.parametrize("n,batch", [(3, 1), (36, 5), (130, 3), (257, 2)])
def test_complex_products(dev, n, batch):
    import torch
    rng = np.random.default_rng(n + batch)
    ld = (n + 7) // 8 * 8
    z = [rng.integers(-2 ** 20, 2 ** 20, (batch, n, n)) + 1j * rng.integers(-2 ** 20, 2 ** 20, (batch, n, n)) for _ in range(3)]
    A, B, D = z[0], z[1], z[2] + np.conj(z[2].transpose(0, 2, 1))
    H = B + np.conj(B.transpose(0, 2, 1))

    def planar(m):
        out = np.full((batch, 2, ld, ld), np.nan)
        out[:, 0, :n, :n], out[:, 1, :n, :n] = m.real, m.imag
        return _cuda(out)

    def back(t):
        t = t.cpu().numpy()[:, :, :n, :n]
        return t[:, 0] + 1j * t[:, 1]

    work = torch.empty(int(dev.crt_complex_bytes(n, batch)), dtype=torch.uint8, device="cuda:0")
    err = torch.zeros(1, dtype=torch.int32, device="cuda:0")
    nan = lambda: torch.full((batch, 2, ld, ld), float("nan"), dtype=torch.float64, device="cuda:0")

    def norms(m):
        return np.sqrt((np.abs(m) ** 2).sum(2))

    def near(got, exact, left, cols, extra=0.0):
        tol = 1.6 * np.sqrt(2 * n) * 2.0 ** -58 * norms(left)[:, :, None] * norms(cols)[:, None, :] + 2.0 ** -50 * (
            np.abs(exact) + np.abs(extra))
        assert np.all(np.abs(got - exact - extra) <= 2 * tol)

    # a general B from the rows of B^T, with the transposed copy
    c, t = nan(), nan()
    Bt = np.ascontiguousarray(B.transpose(0, 2, 1))
    assert dev.crt_complex(_p(planar(A)), _p(planar(Bt)), 0, n, ld, batch, 1.0, 0.0, None, _p(c), _p(t), 0, _p(work), _p(err)) == 0
    torch.cuda.synchronize()
    near(back(c), A @ B, A, Bt)
    assert np.array_equal(back(t), back(c).transpose(0, 2, 1))
    # a Hermitian B from its own rows; a Hermitian result (H H) with D, mirrored with the conjugate
    c = nan()
    assert dev.crt_complex(_p(planar(A)), _p(planar(H)), 1, n, ld, batch, 1.0, 0.0, None, _p(c), None, 0, _p(work), _p(err)) == 0
    torch.cuda.synchronize()
    near(back(c), A @ H, A, H)
    c = planar(D)
    assert dev.crt_complex(_p(planar(H)), _p(planar(H)), 1, n, ld, batch, 1.0, -2.0, _p(c), _p(c), None, 1, _p(work), _p(err)) == 0
    torch.cuda.synchronize()
    near(back(c), H @ H, H, H, -2.0 * D)
    assert np.array_equal(back(c), np.conj(back(c).transpose(0, 2, 1))) and int(err.item()) == 0


def _factor(L, A):
    import torch
    batch, ld = A.shape[:2]
    a = _cuda(A)
    dinv = torch.full((batch, ld // 64, 64, 64), float("nan"), dtype=torch.float64, device="cuda:0")
    work = torch.empty(int(L.crt_cholesky_bytes(C.c_longlong(ld), batch)), dtype=torch.uint8, device="cuda:0")
    status = torch.zeros(1, dtype=torch.int32, device="cuda:0")
    assert L.crt_cholesky(_p(a), C.c_longlong(ld), batch, _p(dinv), _p(work), _p(status)) == 0
    torch.cuda.synchronize()
    return np.tril(a.cpu().numpy()), dinv.cpu().numpy(), int(status.item())


@pytest.mark.parametrize("ld,batch", [(128, 1), (256, 3), (512, 2), (640, 16), (1280, 2)])
def test_cholesky_factors(dev, ld, batch):
    # one and several panels, rows of very different size, poisoned upper halves.  A backward-stable
    # factorisation leaves |A - L L^T|_ij <= (ld + 2) 2^-53 sqrt(A_ii A_jj) and some
    rng = np.random.default_rng(ld)
    dev.crt_cholesky_bytes.restype = C.c_size_t
    A = np.zeros((batch, ld, ld))
    for b in range(batch):
        X = rng.normal(size=(ld, ld)) / np.sqrt(ld)
        d = np.exp(rng.uniform(-4, 4, ld)) if b else np.ones(ld)
        A[b] = (X @ X.T + np.diag(rng.uniform(1e-3, 1.0, ld))) * np.outer(d, d)
    got, dinv, status = _factor(dev, np.where(np.tri(ld, dtype=bool), A, np.nan))
    assert status == 0
    size = np.sqrt(np.einsum("bi,bj->bij", A.diagonal(axis1=1, axis2=2), A.diagonal(axis1=1, axis2=2)))
    back = got @ got.transpose(0, 2, 1)
    assert np.all(np.abs(back - A) <= 2 * (ld + 2) * 2.0 ** -53 * size)
    for b in range(batch):
        for j in range(ld // 64):
            blk = got[b, 64 * j:64 * j + 64, 64 * j:64 * j + 64]
            tol = 8 * 64 * 2.0 ** -53 * (np.abs(dinv[b, j]) @ np.abs(blk))
            assert np.all(np.abs(dinv[b, j] @ blk - np.eye(64)) <= tol + 1e-300)
            assert np.all(np.triu(dinv[b, j], 1) == 0.0)


def test_cholesky_flags_what_is_not_positive_definite(dev):
    dev.crt_cholesky_bytes.restype = C.c_size_t
    rng = np.random.default_rng(9)
    X = rng.normal(size=(640, 640))
    good = X @ X.T + np.eye(640)
    for where in (0, 100, 600):
        for value in (-1.0, 0.0, np.nan):
            A = np.stack([good, good])
            A[1, where, where] = value
            assert _factor(dev, A)[2] == 2   # ST_SCS_NOT_PD
    A = np.stack([good, good])
    A[0, 630, 10] = A[0, 10, 630] = 1e6      # positive diagonal, negative eigenvalue
    assert _factor(dev, A)[2] == 2


def _sunk(rng, ld, row, ratio):
    # positive definite but for one row: L's entries left of the diagonal carry `ratio` times the
    # row's diagonal element, so that its pivot is (1 - ratio) A_rr (the rows below are apart from it)
    X = rng.normal(size=(ld, ld)) / np.sqrt(ld)
    A = X @ X.T + np.diag(rng.uniform(0.1, 1.0, ld))
    L = np.linalg.cholesky(A)
    A[row, row] = (L[row, :row] ** 2).sum() / ratio
    A[row + 1:, :row + 1] = A[:row + 1, row + 1:] = 0.0
    return A


@pytest.mark.parametrize("ld", [128, 256, 512, 640])
def test_cholesky_flags_every_row_longer_than_its_diagonal(dev, ld):
    # a row's scale comes from its diagonal element, which bounds the row of the factor only if the
    # matrix is positive definite: a longer row's product would come back modulo P
    dev.crt_cholesky_bytes.restype = C.c_size_t
    A = np.eye(128)
    A[100, :64] = A[:64, 100] = np.sqrt(2.0 / 64)   # lowest eigenvalue 1 - sqrt(2)
    assert _factor(dev, A[None])[2] == 2
    rng = np.random.default_rng(ld)
    passed = []
    for ratio in np.exp(np.linspace(np.log(1.0 + 1e-6), np.log(10.0), 60)):
        row = int(rng.integers(64, ld))
        A = _sunk(rng, ld, row, ratio)
        if _factor(dev, A[None])[2] != 2:
            passed.append((row, ratio))
    assert not passed


@pytest.mark.parametrize("ld,row", [(128, 64), (128, 127), (640, 600)])
def test_cholesky_keeps_what_is_barely_positive_definite(dev, ld, row):
    dev.crt_cholesky_bytes.restype = C.c_size_t
    A = _sunk(np.random.default_rng(row), ld, row, 1.0 - 1e-9)
    assert np.linalg.cholesky(A)[row, row] > 0.0 and _factor(dev, A[None])[2] == 0


@pytest.mark.parametrize("row,col", [(70, 10), (70, 11), (600, 10), (600, 63), (639, 598)])
def test_cholesky_flags_a_nan_beside_finite_entries(dev, row, col):
    dev.crt_cholesky_bytes.restype = C.c_size_t
    rng = np.random.default_rng(row + col)
    X = rng.normal(size=(640, 640))
    A = X @ X.T + np.eye(640)
    A[row, col] = A[col, row] = np.nan
    assert _factor(dev, A[None])[2] == 2


def _lowest(R, a0, c6, ra, rw, u):
    """Lowest eigenvalue of I + alpha(iu)^(1/2) T^lr alpha(iu)^(1/2) of MBD-NL oscillators."""
    a, om, rad = a0 * ra, 4.0 * c6 / (3.0 * a0 ** 2) * rw, 2.5 * a0 ** (1.0 / 7.0) * ra ** (1.0 / 3.0)
    r = R[None] - R[:, None]
    d = np.sqrt((r ** 2).sum(-1) + np.eye(len(R)))
    f = 1.0 / (1.0 + np.exp(-6.0 * (d / (0.83 * (rad[:, None] + rad[None])) - 1.0)))
    T = np.eye(3) / d[..., None, None] ** 3 - 3.0 * r[..., :, None] * r[..., None, :] / d[..., None, None] ** 5
    al = np.sqrt(a / (1.0 + (u / om) ** 2))
    B = (f * al[:, None] * al[None] * (1.0 - np.eye(len(R))))[..., None, None] * T
    return np.linalg.eigvalsh(np.eye(3 * len(R)) + B.transpose(0, 2, 1, 3).reshape(3 * len(R), -1))[0]


def test_log_energy_refuses_dense_random_oscillators(dev):
    # random positions without a least distance: some I + A_k are not positive definite
    from paper_2308_03140_gb300 import synthetic as syn
    x = np.polynomial.legendre.leggauss(15)[0]
    nodes, seen = 0.6 * (1 + x) / (1 - x), set()
    base = syn.sphere_cluster(74, seed=1)
    with binding.MBD(0, scs_mode=binding.MBD_SCS_NL) as m:
        for seed in range(40):
            rng = np.random.default_rng(seed)
            R = rng.uniform(0, rng.uniform(9.0, 16.0), (74, 3))
            ra, rw = syn.nl_ratios(74, seed)
            m.set_geometry(R)
            m.set_nl_params(base.alpha0_ref, base.c6_ref, ra, rw)
            code = 0
            for call in (lambda: m.evaluate(False), lambda: m.log_energy(1)):
                try:
                    call()
                    code = 0
                except binding.MBDError as e:   # (the energy itself may have no square root)
                    code = e.code
            low = min(_lowest(R, base.alpha0_ref, base.c6_ref, ra, rw, u) for u in nodes)
            assert abs(low) > 1e-9 and code == (0 if low > 0 else 4), (seed, low, code)
            seen.add(code)
    assert seen == {0, 4}
