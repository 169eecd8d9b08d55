"""Epilogue of the wide tensor-core GEMM: every output at one tile, an odd number of tiles and several, the
operand parts to the bit, a transpose that is not 16-byte aligned, and D overwritten in place."""
import pytest

from paper_2308_03140_gb300 import binding

pytestmark = pytest.mark.gpu
TOL = {0: 2e-3, 1: 5e-5, 2: 3e-5}   # per product relative to |A||B|^T (test_gpu_tensorcore.py)


def _operands(n, k, kind, seed):
    import torch
    A = torch.randn(n, k, generator=torch.Generator().manual_seed(seed), dtype=torch.float32).cuda()
    if kind == 0:
        return A, A, None
    if kind == 1:
        hi = A.to(torch.bfloat16)
        return A, hi, (A - hi.float()).to(torch.bfloat16)
    hi = ((A.view(torch.int32) + 0x1000) & ~0x1FFF).view(torch.float32)
    return A, hi, A - hi


def _parts(x, kind):
    """hi and lo of x, each rounded to nearest (TF32: ties away, 10 mantissa bits)."""
    import torch
    if kind == 1:
        hi = x.to(torch.bfloat16)
        return hi, (x - hi.float()).to(torch.bfloat16)
    tf32 = lambda v: ((v.contiguous().view(torch.int32) + 0x1000) & ~0x1FFF).view(torch.float32)
    hi = tf32(x)
    return hi, tf32(x - hi)


@pytest.mark.parametrize("n", [128, 384, 1280])
@pytest.mark.parametrize("kind", [1, 2])
def test_symmetric_product_with_addend_and_parts(kind, n):
    import torch
    k = 192
    A, hi, lo = _operands(n, k, kind, n + kind)
    D = torch.randn(n, n, generator=torch.Generator().manual_seed(3)).cuda()
    D = D + D.T
    C = torch.full_like(D, float("nan"))
    part = torch.bfloat16 if kind == 1 else torch.float32
    H, L = torch.zeros(n, n, dtype=part, device="cuda"), torch.zeros(n, n, dtype=part, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    rc = binding.mbdk_gemm_tc(kind, hi, hi, C, A1=lo, B1=lo, alpha=-0.5, beta=1.5, D=D, C_hi=H, C_lo=L, mode=2, err=err,
                              chunk_stages=2)
    torch.cuda.synchronize()
    assert rc == 0 and err.item() == 0
    assert torch.equal(C, C.T)
    ref = 1.5 * D.double() - 0.5 * A.double() @ A.double().T
    assert (C.double() - ref).abs().max().item() <= TOL[kind] * (A.double().abs() @ A.double().abs().T).max().item()
    h, l = _parts(C, kind)
    assert torch.equal(H, h) and torch.equal(L, l)


@pytest.mark.parametrize("shift", [0, 1, 2])
@pytest.mark.parametrize("kind", [0, 1, 2])
def test_transpose_of_any_alignment(kind, shift):
    import torch
    n, k = 384, 128
    A, hi, lo = _operands(n, k, kind, 7)
    C = torch.full((n, n), float("nan"), device="cuda")
    T = torch.full((n * n + 4,), float("nan"), device="cuda")[shift:shift + n * n].view(n, n)
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    rc = binding.mbdk_gemm_tc(kind, hi, hi, C, A1=lo, B1=lo, CT=T, err=err, chunk_stages=1)
    torch.cuda.synchronize()
    assert rc == 0 and err.item() == 0
    assert torch.equal(T, C.T)
    ref = A.double() @ A.double().T
    assert (C.double() - ref).abs().max().item() <= TOL[kind] * (A.double().abs() @ A.double().abs().T).max().item()


def test_lower_tiles_in_place():
    import torch
    n, k = 640, 256
    A, hi, lo = _operands(n, k, 2, 11)
    C = torch.randn(n, n, generator=torch.Generator().manual_seed(5)).cuda()
    ref = C.double() - A.double() @ A.double().T
    upper = C.clone()
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    rc = binding.mbdk_gemm_tc(2, hi, hi, C, A1=lo, B1=lo, alpha=-1.0, beta=1.0, D=C, mode=1, err=err, chunk_stages=2)
    torch.cuda.synchronize()
    assert rc == 0 and err.item() == 0
    t = torch.arange(n, device="cuda") // 128
    low = t[:, None] >= t[None, :]
    assert torch.equal(C[~low], upper[~low])
    d = (C.double() - ref).abs()[low].max().item()
    assert d <= TOL[2] * (A.double().abs() @ A.double().abs().T).max().item()


@pytest.mark.parametrize("shift", [1, 2, 3])
@pytest.mark.parametrize("kind", [0, 1, 2])
def test_one_symmetric_tile_at_any_address(kind, shift):
    # a tile on the diagonal is stored entry by entry where its outputs do not start on 16 bytes
    import torch
    n, k = 128, 192
    A, hi, lo = _operands(n, k, kind, 21)
    part = torch.bfloat16 if kind == 1 else torch.float32
    at = lambda dtype: torch.zeros(n * n + 4, dtype=dtype, device="cuda")[shift:shift + n * n].view(n, n)
    C, H, L = at(torch.float32), at(part), at(part)
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    rc = binding.mbdk_gemm_tc(kind, hi, hi, C, A1=lo, B1=lo, C_hi=H if kind else None, C_lo=L if kind else None, mode=2, err=err,
                              chunk_stages=1)
    torch.cuda.synchronize()
    assert rc == 0 and err.item() == 0 and torch.equal(C, C.T)
    ref = A.double() @ A.double().T
    assert (C.double() - ref).abs().max().item() <= TOL[kind] * (A.double().abs() @ A.double().abs().T).max().item()
    if kind:
        h, l = _parts(C, kind)
        assert torch.equal(H, h) and torch.equal(L, l)
