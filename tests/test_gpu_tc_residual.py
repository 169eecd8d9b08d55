"""|I - C|^2 of the tensor-core GEMM's epilogue, which ends the Newton-Schulz iteration: as exact as FP64 sums."""
import ctypes as C
import os
import subprocess
from fractions import Fraction

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
    so, libdir = os.path.join(out, "residual_device.so"), os.path.dirname(build.LIB)
    cmd = [build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", f"-I{build.CSRC}",
           os.path.join(HERE, "residual_device.cu"), "-o", so, f"-L{libdir}", f"-l:{os.path.basename(build.LIB)}",
           "-Xlinker", f"-rpath={libdir}"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    L = C.CDLL(so)
    L.tc_residual.argtypes = [C.c_void_p] * 5 + [C.c_int, C.c_int, C.c_void_p, C.c_void_p]
    return L


def residual(L, V, nvalid):
    """Of C = I V^T, exact for a V of TF32 numbers."""
    import torch
    n = V.shape[0]
    t = lambda x: torch.tensor(x, dtype=torch.float32, device="cuda:0")
    eye, zero, v, c = t(np.eye(n)), t(np.zeros((n, n))), t(V.T.copy()), t(np.zeros((n, n)))
    resid = torch.zeros(1, dtype=torch.float64, device="cuda:0")
    err = torch.zeros(1, dtype=torch.int32, device="cuda:0")
    p = lambda x: x.data_ptr()
    torch.cuda.synchronize()
    assert L.tc_residual(p(eye), p(zero), p(v), p(zero), p(c), n, nvalid, p(resid), p(err)) == 0
    torch.cuda.synchronize()
    assert int(err.item()) == 0 and np.array_equal(c.cpu().numpy(), V.astype(np.float32))
    e = np.eye(n) - V
    return resid.item(), sum(Fraction(float(x)) ** 2 for x in e[:nvalid, :nvalid].ravel())


def tf32(x):
    return (np.asarray(x, dtype=np.float32).view(np.uint32) & np.uint32(0xffffe000)).view(np.float32).astype(np.float64)


@pytest.mark.parametrize("n,nvalid", [(128, 128), (128, 70), (384, 300)])
@pytest.mark.parametrize("size", [1.0, 1e-4])
def test_residual_is_as_exact_as_fp64_sums(dev, n, nvalid, size):
    # a thread's sum to far below 2^-53, then at most 5 + 8 + 8 n^2 / 128^2 additions in FP64
    rng = np.random.default_rng(n + nvalid)
    bound = (14 + 8 * (n // 128) ** 2) * 2.0 ** -53
    for V in (np.eye(n) + tf32(size * rng.normal(size=(n, n))) * (1 - np.eye(n)), tf32(np.eye(n) + size * rng.normal(size=(n, n)))):
        got, want = residual(dev, V, nvalid)
        assert abs(Fraction(got) - want) <= bound * want
    # all in the entries of one thread: rows 3, 11, 19, 27 and four columns of every sixteen
    one = np.zeros((n, n))
    one[np.ix_([3, 11, 19, 27], [c for c in range(min(n, nvalid)) if c % 16 // 4 == 1 and c < 128])] = 1.0
    for _ in range(20):
        V = np.eye(n) * (1 - one) + tf32(size * rng.normal(size=(n, n))) * one
        got, want = residual(dev, V, nvalid)
        assert abs(Fraction(got) - want) <= bound * want
