"""The branches that large systems and full cards take, on small systems with small limits: products in panels, the
Cholesky factorisation's trailing updates in groups of matrices and in strips, Bloch vectors in groups and pairs in
chunks, and the kernels on the FP64 pipe that run where the tensor-core products' scratch does not fit."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import oracle as o
from paper_2308_03140_gb300 import binding, build
from paper_2308_03140_gb300 import synthetic as syn
from test_gpu_periodic import small_cell

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
GIB = 1 << 30


@pytest.fixture(scope="module")
def dev():
    build.build()
    binding.load()
    out = os.path.join(HERE, "_build")
    os.makedirs(out, exist_ok=True)
    so = os.path.join(out, "scratch_limits.so")
    libdir = os.path.dirname(build.LIB)
    cmd = [build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", f"-I{build.CSRC}",
           os.path.join(HERE, "scratch_limits.cu"), "-o", so, f"-L{libdir}", f"-l:{os.path.basename(build.LIB)}",
           "-Xlinker", f"-rpath={libdir}"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    L = C.CDLL(so)
    vp, i, sz, ll = C.c_void_p, C.c_int, C.c_size_t, C.c_longlong
    L.limit_context.argtypes = [vp, i, i, sz, i, sz, sz]
    L.limit_context.restype = None
    L.limited_cholesky_bytes.argtypes, L.limited_cholesky_bytes.restype = [ll, i, sz, i], sz
    L.limited_cholesky.argtypes = [vp, ll, i, vp, vp, vp, sz, i]
    return L


def limit(L, calc, none=0, panel=8192, trailing=GIB, strip=2048, cell_products=2 * GIB, cell_sums=GIB):
    L.limit_context(calc.h, none, panel, trailing, strip, cell_products, cell_sums)


def cluster(L, n, **limits):
    s = syn.sphere_cluster(n, seed=1000 + n)
    with binding.MBD(0) as m:
        limit(L, m, **limits)
        m.set_geometry(s.coords)
        m.set_free_atom_params(s.alpha0_ref, s.c6_ref, s.rvdw_ref, s.ratio)
        E, gR, gp, al = m.evaluate(True)
        return dict(E=E, gR=gR, gp=gp, al=al, log=m.log_energy(2)[0], tensor=m.workspace()["tensor_products"])


def near(a, b):
    # both are FP64 to rounding: the bounds of the parity tests against the oracle
    assert abs(a["E"] - b["E"]) <= 1e-10 * abs(b["E"]) and np.allclose(a["al"], b["al"], rtol=1e-11, atol=0)
    assert np.abs(a["gR"] - b["gR"]).max() <= 1e-8
    for x, y in zip(a["gp"], b["gp"]):
        assert np.abs(x - y).max() <= 1e-8 * max(np.abs(y).max(), 1e-3)


@pytest.mark.parametrize("n", [5, 43, 90])
def test_cluster_on_the_fp64_pipe(dev, n):
    a, b = cluster(dev, n, none=1), cluster(dev, n)
    assert not a["tensor"] and b["tensor"]
    near(a, b)
    assert abs(a["log"] - b["log"]) <= 1e-10 * abs(b["log"])


@pytest.mark.parametrize("n", [43, 80, 171])   # order 129: a panel and a column; 240; 513: four panels and a column
def test_newton_schulz_in_panels(dev, n):
    near(cluster(dev, n, panel=128), cluster(dev, n))


@pytest.mark.parametrize("ld,trailing,strip", [(1280, 20_000_000, 2048),    # groups of two matrices and one
                                               (1408, 0, 256),              # strips of 256 columns, the last one shorter
                                               (1152, 0, 256)])
def test_cholesky_in_groups_and_strips(dev, ld, trailing, strip):
    import torch
    rng = np.random.default_rng(ld)
    X = rng.normal(size=(3, ld, ld)) / np.sqrt(ld)
    A = X @ X.transpose(0, 2, 1) + np.stack([np.diag(rng.uniform(0.1, 1.0, ld)) for _ in range(3)])

    def factor(trailing, strip):
        a = torch.tensor(A, device="cuda:0")
        dinv = torch.zeros(3 * (ld // 64) * 4096, dtype=torch.float64, device="cuda:0")
        size = dev.limited_cholesky_bytes(ld, 3, trailing, strip)
        work = torch.empty(size, dtype=torch.uint8, device="cuda:0")
        status = torch.zeros(1, dtype=torch.int32, device="cuda:0")
        p = lambda t: C.c_void_p(t.data_ptr())
        assert dev.limited_cholesky(p(a), ld, 3, p(dinv), p(work), p(status), trailing, strip) == 0
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        return torch.tril(a), dinv, size

    small, whole = factor(trailing, strip), factor(GIB, 2048)
    assert small[2] < whole[2]
    assert torch.equal(small[0], whole[0]) and torch.equal(small[1], whole[1])   # the same products, in other launches
    want = np.linalg.cholesky(A)
    assert np.abs(whole[0].cpu().numpy() - want).max() <= 1e-12 * np.abs(want).max()


def cell(L, N, edge, grid, precision=binding.MBD_PREC_FP64, **limits):
    R, A, p = small_cell(N, edge, 20 + N)
    with binding.MBD(0, precision=precision, ewald_gamma=0.3, real_cutoff=6.5 / 0.3, recip_cutoff=11 * 0.3) as m:
        limit(L, m, **limits)
        m.set_geometry(R, A, grid)
        m.set_free_atom_params(*p)
        E, gR, gp, al = m.evaluate(True)
        return dict(E=E, gR=gR, gp=gp, al=al, gA=m.lattice_gradient(), **m.workspace())


CELLS = [(3, 8.0, (3, 3, 2)), (24, 12.5, (1, 2, 3)), (45, 15.0, (2, 1, 2))]


@pytest.mark.parametrize("N,edge,grid", CELLS)
def test_cell_on_the_fp64_pipe_against_the_oracle(dev, N, edge, grid):
    a = cell(dev, N, edge, grid, none=1)
    assert not a["tensor_products"]
    R, A, p = small_cell(N, edge, 20 + N)
    kap = o.monkhorst_pack(grid)
    E, det = o.periodic_rsscs_energy(R, A, kap, *p, 0.3, 6.5 / 0.3, 11 * 0.3, detail=True)
    _, gR, gA, gp = o.periodic_rsscs_gradient(R, A, kap, *p, 0.3, 6.5 / 0.3, 11 * 0.3)
    near(a, dict(E=E, gR=gR, gp=gp, al=det["alpha_bar"][0]))
    assert np.abs(a["gA"] - gA).max() <= 1e-8


@pytest.mark.parametrize("N,edge,grid", CELLS)
@pytest.mark.parametrize("parts", [dict(cell_products=0, cell_sums=0), dict(cell_products=6_000_000, cell_sums=12_000_000)])
def test_cell_in_groups_and_chunks(dev, N, edge, grid, parts):
    a, b = cell(dev, N, edge, grid, **parts), cell(dev, N, edge, grid)
    assert a["tensor_products"] and b["tensor_products"]
    near(a, b)
    assert abs(a["E"] - b["E"]) <= 1e-13 * abs(b["E"])
    assert np.abs(a["gA"] - b["gA"]).max() <= 1e-10 * np.abs(b["gA"]).max()


@pytest.mark.parametrize("precision", [binding.MBD_PREC_BF16X3, binding.MBD_PREC_TF32X3])
@pytest.mark.parametrize("limits", [dict(none=1), dict(cell_sums=0)])
def test_mixed_cell_one_vector_at_a_time(dev, precision, limits):
    a, b = (cell(dev, 24, 12.5, (2, 2, 2), precision, **l) for l in (limits, {}))
    assert b["matrices_together"] > 1 and a["matrices_together"] == (1 if "none" in limits else b["matrices_together"])
    # every matrix takes its own steps, alone or in a group; the gradient's real-space sums are FP64 either way
    assert abs(a["E"] - b["E"]) <= 1e-12 * abs(b["E"])
    for k in ("gR", "gA", "gp"):
        assert np.abs(np.asarray(a[k]) - np.asarray(b[k])).max() <= 1e-9 * np.abs(np.asarray(b[k])).max()
