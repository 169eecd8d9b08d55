"""The parameter gradient of the learned screening model (mbdk_mlp_backward) at the edges of its blocks of
32 atoms and of their division among eight CTAs, and the training step: the same inputs give the same bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2308_03140_gb300 import binding, build, learned

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    binding.load()


def inputs(B, members, seed):
    rng = np.random.default_rng(seed)
    f = lambda x: torch.tensor(np.asarray(x, dtype=np.float32), device=DEV)
    p = learned.init_params(members, seed + 1) + rng.normal(0.0, 0.01, (members, learned.P)).astype(np.float32)
    X, mean, std = f(rng.normal(0.0, 1.0, (B, learned.F))), f(rng.normal(0.0, 0.1, learned.F)), f(rng.uniform(0.8, 1.2, learned.F))
    return X, mean, std, f(p), f(rng.normal(0.0, 1.0, (B, 16)))


def parts(p):
    cut = np.cumsum([0, learned.F * 128, 128, 128 * 128, 128, 128 * 16, 16])
    W1, b1, W2, b2, W3, b3 = [p[i:j] for i, j in zip(cut, cut[1:])]
    return W1.reshape(learned.F, 128), b1, W2.reshape(128, 128), b2, W3.reshape(128, 16), b3


def gradient(x, z1, z2, dy, W2, W3, mag=lambda v: v):
    """The gradient in FP64 from the cached pre-activations; mag = abs: the sums of the terms' magnitudes."""
    sg = torch.sigmoid
    d = lambda z: mag(sg(z) * (1 + z * (1 - sg(z))))
    h1, h2 = mag(z1 * sg(z1)), mag(z2 * sg(z2))
    d2 = (mag(dy) @ mag(W3).T) * d(z2)
    d1 = (d2 @ mag(W2).T) * d(z1)
    return torch.cat([(mag(x).T @ d1).ravel(), d1.sum(0), (h1.T @ d2).ravel(), d2.sum(0), (h2.T @ mag(dy)).ravel(), mag(dy).sum(0)])


@pytest.mark.parametrize("B", [1, 32, 33, 256, 257, 2100])
def test_parameter_gradient(B):
    # an entry is a sum over atoms of products of two factors; the factors carry the roundings of up to 128 + 16
    # terms and of the activation, the sum those of its 32 + B / 256 + 8 additions: 400 roundings at most of the
    # magnitudes' sum (B <= 2100)
    X, mean, std, p, dY = inputs(B, 2, 40 + B)
    p16 = p.to(torch.float16)
    Y, z = torch.zeros(2, B, 16, device=DEV), torch.zeros(2, 2, B, 128, device=DEV)
    binding.mbdk_mlp_forward(X, mean, std, p16, Y, z)
    dy = torch.stack([dY, dY.flip(0)]).contiguous()
    grad = torch.zeros(2, learned.P, device=DEV)
    binding.mbdk_mlp_backward(X, mean, std, p16, z, dy, None, grad)
    x = (X.double() - mean.double()) / std.double()
    for k in range(2):
        _, _, W2, _, W3, _ = parts(p16[k].double())
        a = (x, z[k, 0].double(), z[k, 1].double(), dy[k].double(), W2, W3)
        err, size = (grad[k].double() - gradient(*a)).abs(), gradient(*a, mag=torch.abs)
        assert bool((err <= 400 * 2.0 ** -24 * size).all()), float((err / size).max())
    first = grad.clone()
    binding.mbdk_mlp_backward(X, mean, std, p16, z, dy, torch.zeros(2, B, learned.F, device=DEV), grad)
    assert torch.equal(grad, 2 * first)   # accumulated; the same with dX


@pytest.mark.parametrize("B", [100, 4096])
def test_training_steps_repeat_to_the_bit(B):
    X, mean, std, p0, T = inputs(B, 2, B)

    def steps():
        p, p16, grad = p0.clone(), p0.to(torch.float16), torch.zeros_like(p0)
        m, v = torch.zeros_like(p0), torch.zeros_like(p0)
        Y, dY, z = torch.zeros(2, B, 16, device=DEV), torch.zeros(2, B, 16, device=DEV), torch.zeros(2, 2, B, 128, device=DEV)
        loss = torch.zeros(2, dtype=torch.float64, device=DEV)
        for step in (1, 2, 3):
            grad.zero_()
            binding.mbdk_mlp_forward(X, mean, std, p16, Y, z)
            for k in range(2):
                binding.mbdk_mse_grad(Y[k], T, dY[k], loss[k:k + 1])
            binding.mbdk_mlp_backward(X, mean, std, p16, z, dY, None, grad)
            binding.mbdk_adam_step(p, grad, m, v, step, 2e-3, p16)
        return grad, p, m, v, p16, Y, loss

    a = steps()
    for _ in range(5):
        b = steps()
        for x, y in zip(a[:-1], b[:-1]):
            assert torch.equal(x, y)
        # (the loss is summed by FP64 atomics of positive terms)
        assert bool(((a[-1] - b[-1]).abs() <= 16 * B * 2.0 ** -53 * a[-1]).all())


def test_gradient_on_two_streams_and_from_a_graph():
    # the scratch is the stream's own: calls that overlap, and a captured call, give what one call gives
    X, mean, std, p, dY = inputs(3000, 1, 5)
    p16, dy = p.to(torch.float16), dY[None].contiguous()
    Y, z = torch.zeros(1, 3000, 16, device=DEV), torch.zeros(1, 2, 3000, 128, device=DEV)
    binding.mbdk_mlp_forward(X, mean, std, p16, Y, z)
    grads = [torch.zeros(1, learned.P, device=DEV) for _ in range(3)]
    back = lambda g: binding.mbdk_mlp_backward(X, mean, std, p16, z, dy, None, g)
    back(grads[0])
    torch.cuda.synchronize()
    for _ in range(20):
        for g in grads[1:]:
            g.zero_()
        torch.cuda.synchronize()
        for st, g in zip((torch.cuda.Stream(), torch.cuda.Stream()), grads[1:]):
            with torch.cuda.stream(st):
                back(g)
        torch.cuda.synchronize()
        assert torch.equal(grads[0], grads[1]) and torch.equal(grads[0], grads[2])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        back(grads[1])
    for _ in range(3):
        grads[1].zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(grads[0], grads[1])
