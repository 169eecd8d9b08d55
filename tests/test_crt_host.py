"""The residue arithmetic of the FP64 products on the tensor cores (csrc/crt64.cuh), compiled for
the host (tests/crt_host.cu), against Python's integers: residues, running sums and stored bytes
are exact and stay in the ranges that keep every FP32 sum exact, and the way back returns the
product.  CPU only; the kernels are checked in test_gpu_crt.py."""
import ctypes as C
import math
import os
import subprocess

import numpy as np
import pytest

from paper_2308_03140_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2308_03140_gb300", "csrc")


@pytest.fixture(scope="module")
def host():
    out = os.path.join(HERE, "_build")
    os.makedirs(out, exist_ok=True)
    so = os.path.join(out, "crt_host.so")
    src = os.path.join(HERE, "crt_host.cu")
    if not os.path.exists(so) or any(os.path.getmtime(d) > os.path.getmtime(so)
                                     for d in (src, os.path.join(CSRC, "crt64.cuh"))):
        cmd = [build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", f"-I{CSRC}", src,
               "-o", so]
        res = subprocess.run(cmd, capture_output=True, text=True)
        assert res.returncode == 0, res.stderr
    L = C.CDLL(so)
    L.crt_exponent.argtypes, L.crt_result.restype = [C.c_double], C.c_double
    return L


def ptr(a):
    return a.ctypes.data_as(C.c_void_p)


def moduli(L):
    m = np.zeros(64, dtype=np.int32)
    return m[:L.crt_moduli(ptr(m))].tolist()


def residues(L, x):
    x = np.ascontiguousarray(x, dtype=np.int64)
    r = np.zeros((len(moduli(L)), x.size), dtype=np.float32)
    L.crt_residues(ptr(x), x.size, ptr(r))
    return r


def test_moduli_are_coprime_and_their_product_holds_the_scaled_rows(host):
    m = moduli(host)
    assert all(math.gcd(a, b) == 1 for i, a in enumerate(m) for b in m[:i])
    root = math.sqrt(math.prod(m) / 2)
    for norm in (1.0, 0.65, 0.651, 0.6499999, 3.0, 1e-280, 7e250, math.nextafter(1.0, 2.0), 5e-324):
        e = host.crt_exponent(norm)
        assert root / 3 < math.ldexp(norm, e) < 0.999 * root
    assert host.crt_exponent(0.0) == 0
    assert host.crt_exponent(math.inf) == host.crt_exponent(math.nan) == 0x7fffffff


def test_residues_are_exact_and_small(host):
    rng = np.random.default_rng(1)
    x = np.concatenate([rng.integers(-2 ** 59, 2 ** 59, 4000), rng.integers(-70000, 70000, 4000),
                        [0, 1, -1, 2 ** 59, -2 ** 59, 2 ** 15, -2 ** 15, 2 ** 31, 2 ** 47, -2 ** 47, 2 ** 15 + 2 ** 31 + 2 ** 47]])
    for mi, r in zip(moduli(host), residues(host, x)):
        assert np.all(r == np.rint(r)) and np.all(np.abs(r) <= 128)   # bf16 integers; 1024 products <= 2^24
        assert np.all((r.astype(np.int64) - x) % mi == 0)
        assert np.all((r.view(np.uint32) & 0xffff) == 0)              # exact in bf16


def test_running_sums_and_bytes(host):
    rng = np.random.default_rng(2)
    top = host.crt_chunk() * 128 * 128
    assert top <= 2 ** 24
    v = np.concatenate([rng.integers(-top, top + 1, 5000), [top, -top, 0]]).astype(np.float32)
    for i, mi in enumerate(moduli(host)):
        out = np.zeros_like(v)
        host.crt_reduce(i, ptr(v), v.size, ptr(out))
        assert np.all((out.astype(np.int64) - v.astype(np.int64)) % mi == 0) and np.all(np.abs(out) <= mi / 2 + 1)
        r = np.arange(-mi // 2 - 1, mi // 2 + 2).astype(np.float32)
        y = np.zeros_like(r)
        host.crt_stored(i, ptr(r), r.size, ptr(y))
        rest = math.prod(moduli(host)) // mi
        assert np.all((y >= 0) & (y < mi))
        assert np.all((y.astype(np.int64) * (rest % mi) - r.astype(np.int64)) % mi == 0)


@pytest.mark.parametrize("K", [1, 3, 40, 1500])
def test_products_come_back(host, K):
    # the whole way on rows of the largest norm allowed, against exact integers
    rng = np.random.default_rng(K)
    m = moduli(host)
    P = math.prod(m)
    a, b = rng.normal(size=(6, K)), rng.normal(size=(5, K))
    a[0], a[1, 0], a[5] = 0.0, 1e4, 0.0
    a[5, 0] = b[0, 0] = 1.0
    b[0, 1:] = 0.0                               # a[5].b[0]: two rows of one entry each, the largest product
    ex = [[np.rint(np.ldexp(r, host.crt_exponent(float(np.linalg.norm(r))))).astype(np.int64) for r in s] for s in (a, b)]
    xa, xb = np.array(ex[0]), np.array(ex[1])
    ra, rb = residues(host, xa.ravel()).reshape(len(m), 6, K), residues(host, xb.ravel()).reshape(len(m), 5, K)
    y = np.zeros((len(m), 30), dtype=np.uint8)
    for i, mi in enumerate(m):
        t = (ra[i].astype(np.int64) @ rb[i].astype(np.int64).T) % mi
        t = np.where(2 * t > mi, t - mi, t).astype(np.float32).ravel()
        o = np.zeros_like(t)
        host.crt_stored(i, ptr(t), t.size, ptr(o))
        y[i] = o
    frac = np.zeros(30, dtype=np.int64)
    scale = host.crt_result(ptr(y), 30, ptr(frac))
    assert abs(scale * 2.0 ** 64 - P) <= P * 2.0 ** -52
    for k, f in enumerate(frac):
        exact = sum(int(p) * int(q) for p, q in zip(xa[k // 5], xb[k % 5]))
        assert abs(int(f) * P - (exact << 64)) <= 2 * P   # within two units of the 64-bit fraction
