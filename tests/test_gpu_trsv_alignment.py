"""The triangular solves (mbdk_chol_solve3_f64) on factors that start at any entry of a buffer, and captured in a
graph: the same bits as on an aligned factor."""
import pytest

torch = pytest.importorskip("torch")

from paper_2308_03140_gb300 import binding, build

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    binding.load()


def factor(ld, batch):
    g = torch.Generator().manual_seed(ld)
    X = torch.randn(batch, ld, ld, generator=g, dtype=torch.float64)
    L = (X @ X.transpose(1, 2) / ld + torch.eye(ld, dtype=torch.float64)).to(DEV).contiguous()
    dinv = torch.zeros(batch * (ld // 64) * 4096, dtype=torch.float64, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    binding.mbdk_cholesky_f64(L, dinv, status)
    assert int(status.item()) == 0
    return L, dinv, torch.randn(batch, ld, 3, generator=g, dtype=torch.float64).to(DEV)


@pytest.mark.parametrize("ld,batch", [(64, 1), (128, 3), (640, 2)])
@pytest.mark.parametrize("offset", [1, 2, 3])
def test_solve_with_a_factor_at_any_entry(ld, batch, offset):
    L, dinv, B = factor(ld, batch)
    want = B.clone()
    binding.mbdk_chol_solve3_f64(L, dinv, want)
    buffer = torch.full((L.numel() + offset,), float("nan"), dtype=torch.float64, device=DEV)
    view = buffer[offset:].view(batch, ld, ld)
    view.copy_(L)
    assert view.data_ptr() % 16 == 8 * (offset % 2)
    got = B.clone()
    binding.mbdk_chol_solve3_f64(view, dinv, got)
    assert torch.equal(got, want)


def test_solve_from_a_graph():
    L, dinv, B = factor(640, 2)
    want, got = B.clone(), B.clone()
    binding.mbdk_chol_solve3_f64(L, dinv, want)
    work = torch.zeros_like(B)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        binding.mbdk_chol_solve3_f64(L, dinv, got, work)
    for _ in range(3):
        got.copy_(B)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(got, want)
