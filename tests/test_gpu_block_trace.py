"""The traces of the diagonal blocks of Q^{1/2} (k_block_trace_sqrt) to the bit: they end as right-hand sides of FP32
solves, where a last-place difference would turn a rounding and move the forces by far more than itself."""
import ctypes as C
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_2308_03140_gb300 import binding, build

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))   # rounded once


def traces(V, W, N, sqrt_s):
    """A warp per atom: lane l adds its products k = l, l + 32, ... of rows 3i, 3i + 1, 3i + 2 one row after another."""
    ld, out = V.shape[0], []
    for i in range(N):
        acc = [0.0] * 32
        for p in (3 * i, 3 * i + 1, 3 * i + 2):
            for k in range(ld):
                acc[k % 32] = fma(V[p, k], W[k, p], acc[k % 32])
        for o in (16, 8, 4, 2, 1):
            acc = [acc[l] + acc[l ^ o] for l in range(32)]
        trv = V[3 * i, 3 * i] + V[3 * i + 1, 3 * i + 1] + V[3 * i + 2, 3 * i + 2]
        out.append(sqrt_s * 0.5 * fma(3.0, trv, -acc[0]))
    return np.array(out)


@pytest.mark.parametrize("N", [1, 5, 42])
def test_block_traces_to_the_bit(N):
    import torch
    build.build()
    binding.load()
    out = os.path.join(HERE, "_build")
    os.makedirs(out, exist_ok=True)
    so, libdir = os.path.join(out, "trace_device.so"), os.path.dirname(build.LIB)
    cmd = [build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", f"-I{build.CSRC}",
           os.path.join(HERE, "trace_device.cu"), "-o", so, f"-L{libdir}", f"-l:{os.path.basename(build.LIB)}",
           "-Xlinker", f"-rpath={libdir}"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    L = C.CDLL(so)
    L.block_traces.argtypes = [C.c_void_p, C.c_void_p, C.c_longlong, C.c_int, C.c_double, C.c_void_p]
    rng = np.random.default_rng(N)
    V, W = rng.normal(size=(2, 128, 128))
    v, w, tq = (torch.tensor(x, device="cuda:0") for x in (V, W, np.zeros(N)))
    torch.cuda.synchronize()
    L.block_traces(v.data_ptr(), w.data_ptr(), 128, N, 1.7, tq.data_ptr())
    torch.cuda.synchronize()
    assert np.array_equal(tq.cpu().numpy(), traces(V, W, N, 1.7))
