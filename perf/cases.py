"""The work this library is timed on: energies and gradients of clusters and cells through its
public calls, over the range of sizes, arithmetics and methods it offers, and one training step
of the learned screening model.

A case is a dict of plain values.  `kind` says which program it stands for:

  host      a program with host arrays: new geometry and parameters, then energy, forces,
            parameter gradients (and the lattice gradient of a cell) every step
  device    a program that keeps its tensors on the GPU (mbd_evaluate_dev)
  autograd  a PyTorch program: forward and backward of autograd.MBDEnergy
  ts        the pairwise TS energy with its gradients, host arrays
  train     one optimisation step of the learned screening ensemble, as learned.Ensemble.fit does it

Geometries and parameters are those of synthetic.py (the shapes of the benchmark's workloads).
exact() evaluates the method's formulas in plain torch FP64 and takes derivatives by autograd.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

from paper_2308_03140_gb300 import binding, learned
from paper_2308_03140_gb300 import synthetic as syn
from paper_2308_03140_gb300.autograd import MBDEnergy

PRECISION = {"fp64": binding.MBD_PREC_FP64, "tf32x3": binding.MBD_PREC_TF32X3, "bf16x3": binding.MBD_PREC_BF16X3}
BETA, STEEP, S_R = 0.83, 6.0, 0.94
MEMBERS = 4          # ensemble members of the learned model
TRAIN_STEP = 100     # the optimiser is in the middle of its run
LR = 2e-3


def listed():
    return [
        # A small molecule in the default arithmetic: one step of a geometry optimisation driven
        # from host arrays.  Launches and latency.
        {"name": "mol32_fp64", "kind": "host", "n": 32, "precision": "fp64", "scs": "plain"},
        # A cluster of the batch recipe's middle size in the default arithmetic, from PyTorch.
        {"name": "cluster251_fp64", "kind": "autograd", "n": 251, "precision": "fp64", "scs": "plain"},
        # A large cluster in the default arithmetic, tensors on the GPU.
        {"name": "cluster1000_fp64", "kind": "device", "n": 1000, "precision": "fp64", "scs": "plain"},
        # A molecular crystal's cell in the default arithmetic with all gradients.
        {"name": "cell96_fp64", "kind": "host", "n": 96, "k": 4, "precision": "fp64", "scs": "plain"},
        # The batch's ordinary cluster in the reduced-precision arithmetic.
        {"name": "cluster270_bf16x3", "kind": "autograd", "n": 270, "precision": "bf16x3", "scs": "plain"},
        # The benchmark's 2000-atom cluster.
        {"name": "cluster2000_bf16x3", "kind": "device", "n": 2000, "precision": "bf16x3", "scs": "plain"},
        # The largest cluster whose working set fits the card three times.
        {"name": "cluster5000_bf16x3", "kind": "device", "n": 5000, "precision": "bf16x3", "scs": "plain"},
        # The benchmark's periodic cell: 256 atoms, 64 Bloch vectors, reduced precision.
        {"name": "cell256_bf16x3", "kind": "host", "n": 256, "k": 4, "precision": "bf16x3", "scs": "plain"},
        # MBD-NL (no screening) of a mid-sized cluster in the more accurate reduced precision.
        {"name": "nl1501_tf32x3", "kind": "device", "n": 1501, "precision": "tf32x3", "scs": "nl"},
        # The learned screening on an ordinary cluster: energy and forces.
        {"name": "learned270_bf16x3", "kind": "device", "n": 270, "precision": "bf16x3", "scs": "learned"},
        # TS pairwise energies, the cheap companion of every MBD run.
        {"name": "ts2000", "kind": "ts", "n": 2000},
        # Training the learned screening: one step of the four members at the default batch.
        {"name": "train4096", "kind": "train", "n": 4096},
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    pick = rng.random()
    if pick < 0.35:   # the default arithmetic, small molecules to large clusters
        return {"kind": rng.choice(["host", "device", "autograd"]), "n": _size(rng, 24, 960), "precision": "fp64",
                "scs": rng.choice(["plain", "plain", "plain", "nl"])}
    if pick < 0.5:    # cells in the default arithmetic
        return {"kind": "host", "n": _size(rng, 12, 96), "k": rng.choice([2, 3, 4]), "precision": "fp64", "scs": "plain"}
    if pick < 0.75:   # clusters in the reduced precisions
        return {"kind": rng.choice(["host", "device", "autograd"]), "n": _size(rng, 50, 4500),
                "precision": rng.choice(["bf16x3", "bf16x3", "tf32x3"]), "scs": rng.choice(["plain", "plain", "nl"])}
    if pick < 0.83:   # cells in the reduced precisions
        return {"kind": "host", "n": _size(rng, 48, 240), "k": rng.choice([2, 3, 4]), "precision": "bf16x3",
                "scs": "plain"}
    if pick < 0.9:
        return {"kind": "device", "n": _size(rng, 50, 500), "precision": "bf16x3", "scs": "learned"}
    if pick < 0.95:
        return {"kind": "ts", "n": _size(rng, 100, 4000)}
    return {"kind": "train", "n": _size(rng, 512, 8192)}


# ---- inputs -----------------------------------------------------------------------------
def _system(case, seed):
    """Host arrays of the case: coords, the four parameter arrays, lattice, k-grid."""
    n, s = case["n"], 10_000 + int(seed)
    if "k" in case:   # the benchmark cell's density at any number of atoms
        f = (n / 256.0) ** (1.0 / 3.0)
        sysm = syn.triclinic_cell(n, edge=(20.0 * f, 26.0 * f), k_grid=(case["k"],) * 3, seed=s)
    elif case.get("kind") == "host" and n <= 64:
        sysm = syn.cube_cluster(n, 14.0 * (n / 32.0) ** (1.0 / 3.0), 2.5, seed=s)
    else:
        sysm = syn.sphere_cluster(n, seed=s)
    par = [sysm.alpha0_ref, sysm.c6_ref, sysm.rvdw_ref, sysm.ratio]
    if case.get("scs") == "nl":
        par[2], par[3] = syn.nl_ratios(n, s)
    return sysm.coords, par, sysm.lattice, sysm.k_grid


def _ewald(case):
    """The benchmark cell's explicit Ewald split for large cells, the automatic one for small."""
    return {"ewald_gamma": 0.2, "real_cutoff": 30.0, "recip_cutoff": 2.0} if case["n"] > 128 else {}


def _train_data(case, seed):
    """A training set of twice the batch with features and targets of the size and spread the
    library's own have, and the optimiser's state in the middle of a run."""
    g = np.random.default_rng(20_000 + int(seed))
    n, F, P = case["n"], learned.F, learned.P
    X = g.normal(0.0, 1.0, (2 * n, F)).astype(np.float32)
    Y = (-0.05 + 0.04 * np.tanh(X[:, :16]) + g.normal(0.0, 0.005, (2 * n, 16))).astype(np.float32)
    p = learned.init_params(MEMBERS, int(seed) + 1) + g.normal(0.0, 0.01, (MEMBERS, P)).astype(np.float32)
    m = g.normal(0.0, 1e-4, (MEMBERS, P)).astype(np.float32)
    v = (g.uniform(0.5, 2.0, (MEMBERS, P)) * 1e-7).astype(np.float32)
    mean = (0.1 * g.normal(size=F)).astype(np.float32)
    std = g.uniform(0.8, 1.2, F).astype(np.float32)
    idx = g.integers(0, 2 * n, (MEMBERS, n)).astype(np.int32)
    return X, Y, p, m, v, mean, std, idx


class _State:
    pass


def prepare(case, seed):
    st = _State()
    st.case = case
    dev = torch.device("cuda:0")
    if case["kind"] == "train":
        X, Y, p, m, v, mean, std, idx = [torch.tensor(x, device=dev) for x in _train_data(case, seed)]
        n = case["n"]
        f32 = dict(dtype=torch.float32, device=dev)
        st.X, st.Y, st.p, st.m, st.v, st.mean, st.std, st.idx = X, Y, p, m, v, mean, std, idx
        st.p16, st.grad = p.to(torch.float16), torch.zeros_like(p)
        st.Xb, st.Yb = torch.zeros(n, learned.F, **f32), torch.zeros(n, 16, **f32)
        st.Yp, st.dY = torch.zeros(MEMBERS, n, 16, **f32), torch.zeros(MEMBERS, n, 16, **f32)
        st.z = torch.zeros(MEMBERS, 2, n, 128, **f32)
        st.loss = torch.zeros(MEMBERS, dtype=torch.float64, device=dev)
        st.step = TRAIN_STEP
        return st
    st.coords, st.par, st.lattice, st.k_grid = _system(case, seed)
    if case["kind"] == "ts":
        st.calc = binding.MBD(0)
        st.calc.set_geometry(st.coords)
        return st
    opts = {"precision": PRECISION[case["precision"]]}
    if "k" in case:
        opts.update(_ewald(case))
    if case["scs"] == "nl":
        opts["scs_mode"] = binding.MBD_SCS_NL
    if case["scs"] == "learned":   # no fallback: the model's own energy and forces
        opts.update(scs_mode=binding.MBD_SCS_LEARNED, learned_max_error=1e300)
    if case["kind"] == "autograd":
        st.module = MBDEnergy(case["n"], **opts)
        st.ins = [torch.tensor(x, dtype=torch.float64, device=dev, requires_grad=True) for x in (st.coords, *st.par)]
        return st
    st.calc = binding.MBD(0, **opts)
    if case["scs"] == "learned":
        path = os.path.join(os.path.dirname(os.path.abspath(binding.__file__)), "learned_scs_model.npz")
        with np.load(path) as d:
            st.calc.set_scs_model(d["params16"], d["mean"], d["std"])
    st.calc.set_geometry(st.coords, st.lattice, st.k_grid)
    if case["kind"] == "device":
        n = case["n"]
        f64 = dict(dtype=torch.float64, device=dev)
        st.ins = [torch.tensor(x, **f64) for x in (st.coords, *st.par)]
        st.energy, st.grad_r, st.alpha = torch.empty(1, **f64), torch.empty(n, 3, **f64), torch.empty(n, **f64)
        st.grad_p = None if case["scs"] == "learned" else torch.empty(4, n, **f64)
    return st


def run(st):
    kind = st.case["kind"]
    if kind == "host":
        st.calc.set_geometry(st.coords, st.lattice, st.k_grid)
        st.calc.set_free_atom_params(*st.par)
        E, gR, gp, alpha = st.calc.evaluate(True)
        out = {"energy": E, "grad_coords": gR, "grad_params": gp, "alpha": alpha}
        if st.lattice is not None:
            out["grad_lattice"] = st.calc.lattice_gradient()
        return out
    if kind == "device":
        st.calc.evaluate_dev(*st.ins, st.energy, st.grad_r, st.grad_p, st.alpha)
        out = {"energy": st.energy, "grad_coords": st.grad_r, "alpha": st.alpha}
        if st.grad_p is not None:
            out["grad_params"] = st.grad_p
        return out
    if kind == "autograd":
        E = st.module(*st.ins)
        g = torch.autograd.grad(E, st.ins)
        return {"energy": E.detach(), "grad_coords": g[0], "grad_params": list(g[1:])}
    if kind == "ts":
        st.calc.set_geometry(st.coords)
        st.calc.set_free_atom_params(*st.par)
        E, gR, gp = st.calc.ts_energy(S_R)
        return {"energy": E, "grad_coords": gR, "grad_params": gp}
    st.grad.zero_()
    for k in range(MEMBERS):
        binding.mbdk_gather_rows(st.idx[k], st.X, st.Xb)
        binding.mbdk_gather_rows(st.idx[k], st.Y, st.Yb)
        pk = st.p16[k:k + 1]
        binding.mbdk_mlp_forward(st.Xb, st.mean, st.std, pk, st.Yp[k:k + 1], st.z[k:k + 1])
        binding.mbdk_mse_grad(st.Yp[k], st.Yb, st.dY[k], st.loss[k:k + 1])
        binding.mbdk_mlp_backward(st.Xb, st.mean, st.std, pk, st.z[k:k + 1], st.dY[k:k + 1], None, st.grad[k:k + 1])
    binding.mbdk_adam_step(st.p, st.grad, st.m, st.v, st.step, LR, st.p16)
    st.step += 1
    return {"loss": st.loss, "outputs": st.Yp, "grad": st.grad, "params": st.p, "m": st.m, "v": st.v}


# ---- the least work ---------------------------------------------------------------------
def work(case):
    """Inputs and outputs once, and the method's own operations: one factorisation of each of the
    16 screening matrices, about 9 n^3 for the spectrum and inverse root of each
    coupled-oscillator matrix (four times that for a complex one), 60 operations per ordered pair for
    TS, and the products of the network's forward and backward passes."""
    n = case["n"]
    if case["kind"] == "train":
        params = learned.P
        return {"bytes": MEMBERS * (n * (learned.F + 16 + 1 + 16) * 4.0 + params * 4.0 * 8),
                "flops": MEMBERS * n * 6.0 * (learned.F * 128 + 128 * 128 + 128 * 16)}
    io = 8.0 * n * (7 + 3 + 4 + 1)
    if case["kind"] == "ts":
        return {"bytes": io, "flops": 60.0 * n * n}
    order = 3.0 * n
    spectra = 4 * case["k"] ** 3 if "k" in case else 1
    screening = 16 * order ** 3 / 3 if case["scs"] == "plain" else 0.0
    return {"bytes": io, "flops": screening + 9.0 * spectra * order ** 3}


# ---- the same in plain FP64 -------------------------------------------------------------
def _device():
    return torch.device("cuda:0" if torch.cuda.is_available() else "cpu")


def _fermi(d, S, beta, a):
    return 1.0 / (1.0 + torch.exp(-a * (d / (beta * S) - 1.0)))


def _grid():
    x, w = np.polynomial.legendre.leggauss(15)
    return np.concatenate([[0.0], 0.6 * (1 + x) / (1 - x)]), np.concatenate([[0.0], 1.2 / (1 - x) ** 2 * w])


def _screened(alpha_of_block, a0, om, rv):
    """Screened alpha(0), omega and R_vdW; alpha_of_block(alpha(u)) is the screened alpha(u)."""
    u, w = _grid()
    rows = [alpha_of_block(a0 / (1.0 + (uk / om) ** 2)) for uk in u]
    c6 = 3.0 / math.pi * sum(wk * r * r for wk, r in zip(w[1:], rows[1:]))
    return rows[0], 4.0 / 3.0 * c6 / rows[0] ** 2, rv * (rows[0] / a0) ** (1.0 / 3.0)


def _gauss_tensor(r, d, alpha):
    """T^GG between oscillators of polarizability alpha at r (.., n, n, 3), d = |r|."""
    sig = (math.sqrt(2.0 / math.pi) / 3.0 * alpha) ** (1.0 / 3.0)
    z = d / torch.sqrt(sig[:, None] ** 2 + sig[None, :] ** 2)
    th = 2.0 / math.sqrt(math.pi) * z * torch.exp(-z * z)
    F = torch.erf(z) - th
    eye = torch.eye(3, dtype=r.dtype, device=r.device)
    return (F / d ** 3)[..., None, None] * eye + ((2 * z * z * th - 3 * F) / d ** 5)[..., None, None] * (
        r[..., :, None] * r[..., None, :])


def _bare(r, d):
    eye = torch.eye(3, dtype=r.dtype, device=r.device)
    return eye / d[..., None, None] ** 3 - 3.0 * r[..., :, None] * r[..., None, :] / d[..., None, None] ** 5


def _blocks(T):
    n = T.shape[0]
    return T.permute(0, 2, 1, 3).reshape(3 * n, 3 * n)


def _solve_alpha(alpha, B):
    n = alpha.shape[0]
    E = torch.eye(3, dtype=B.dtype, device=B.device).repeat(n, 1)
    X = torch.linalg.solve(torch.diag((1.0 / alpha).repeat_interleave(3)) + B, E)
    return X.reshape(n, 3, 3).diagonal(dim1=1, dim2=2).sum(1) / 3.0


def _exact_cluster(case, coords, par):
    dev = _device()
    R, p0, p1, p2, p3 = ins = [torch.tensor(x, dtype=torch.float64, device=dev, requires_grad=True)
                               for x in (coords, *par)]
    n = R.shape[0]
    self_ = torch.eye(n, dtype=torch.bool, device=dev)
    r = R[None, :, :] - R[:, None, :]
    d = torch.where(self_, torch.ones((), dtype=R.dtype, device=dev), (r * r).sum(-1)).sqrt()
    off = (~self_).to(R.dtype)
    if case["scs"] == "nl":
        a, om, rad = p0 * p2, 4.0 * p1 / (3.0 * p0 ** 2) * p3, 2.5 * p0 ** (1.0 / 7.0) * p2 ** (1.0 / 3.0)
    else:
        a0, om0, rv = p0 * p3, 4.0 * p1 / (3.0 * p0 ** 2), p2 * p3 ** (1.0 / 3.0)
        sr = (1.0 - _fermi(d, rv[:, None] + rv[None, :], BETA, STEEP)) * off
        a, om, rad = _screened(lambda al: _solve_alpha(al, _blocks(sr[..., None, None] * _gauss_tensor(r, d, al))),
                               a0, om0, rv)
    g = _fermi(d, rad[:, None] + rad[None, :], BETA, STEEP) * off
    c = om * a.sqrt()
    Q = _blocks((c[:, None] * c[None, :] * g)[..., None, None] * _bare(r, d))
    Q = Q + torch.diag((om * om).repeat_interleave(3))
    E = 0.5 * torch.linalg.eigvalsh(Q).sqrt().sum() - 1.5 * om.sum()
    grads = torch.autograd.grad(E, ins)
    return E.detach(), grads, a.detach()


def _images(A, coords, rc):
    """Every lattice translation (integers [m, 3]) that brings some pair within rc."""
    An = A.detach().cpu().numpy()
    span = np.abs(coords @ np.linalg.inv(An)).max()
    reach = np.ceil(rc * np.linalg.norm(np.linalg.inv(An), axis=0) + 2 * span + 1).astype(int)
    ns = np.stack(np.meshgrid(*[np.arange(-m, m + 1) for m in reach], indexing="ij"), -1).reshape(-1, 3)
    far = np.linalg.norm(coords[None] - coords[:, None], axis=-1).max()
    return ns[np.linalg.norm(ns @ An, axis=1) < rc + far]


def _exact_cell(case, coords, par, lattice, k_grid):
    dev = _device()
    f64 = dict(dtype=torch.float64, device=dev)
    R, p0, p1, p2, p3, A = ins = [torch.tensor(x, requires_grad=True, **f64) for x in (coords, *par, lattice)]
    n = R.shape[0]
    vol0 = abs(float(np.linalg.det(lattice)))
    opt = _ewald(case)
    gam = opt.get("ewald_gamma", 2.5 / vol0 ** (1.0 / 3.0))
    rc, kc = opt.get("real_cutoff", 6.0 / gam), opt.get("recip_cutoff", 10.0 * gam)
    # the pairs (i, j, n) with 0 < |R_j + nA - R_i| < rc
    ns = _images(A, coords, rc)
    base = coords[None, :, :] - coords[:, None, :]
    pi, pj, pn = [], [], []
    for t in ns:
        dist = np.linalg.norm(base + t @ lattice, axis=-1)
        i, j = np.nonzero((dist < rc) & (dist > 1e-8))
        pi.append(i), pj.append(j), pn.append(np.repeat(t[None], len(i), 0))
    pi, pj = (torch.tensor(np.concatenate(x), device=dev) for x in (pi, pj))
    pn = torch.tensor(np.concatenate(pn), **f64)

    def pairs():
        r = R[pj] - R[pi] + pn @ A
        return r, (r * r).sum(-1).sqrt()

    def summed(T):   # sum the pair blocks into the matrix
        return _blocks(torch.zeros(n * n, 3, 3, dtype=T.dtype, device=dev).index_add(0, pi * n + pj, T).reshape(n, n, 3, 3))

    a0, om0, rv = p0 * p3, 4.0 * p1 / (3.0 * p0 ** 2), p2 * p3 ** (1.0 / 3.0)
    r, d = pairs()
    sr = 1.0 - _fermi(d, rv[pi] + rv[pj], BETA, STEEP)
    eye = torch.eye(3, **f64)

    def screened_alpha(al):
        sig = (math.sqrt(2.0 / math.pi) / 3.0 * al) ** (1.0 / 3.0)
        z = d / torch.sqrt(sig[pi] ** 2 + sig[pj] ** 2)
        th = 2.0 / math.sqrt(math.pi) * z * torch.exp(-z * z)
        F = torch.erf(z) - th
        T = (sr * F / d ** 3)[:, None, None] * eye + (sr * (2 * z * z * th - 3 * F) / d ** 5)[:, None, None] * (
            r[:, :, None] * r[:, None, :])
        return _solve_alpha(al, summed(T))

    scr = _screened(screened_alpha, a0, om0, rv)
    a, om, rad = leaf = [x.detach().requires_grad_(True) for x in scr]
    # sum over the Bloch vectors, one backward pass each
    kap = np.array([[(2.0 * m - k - 1) / (2.0 * k) for m in range(1, k + 1)] for k in k_grid])
    grid = [(x, y, z) for x in kap[0] for y in kap[1] for z in kap[2]]
    Bn = 2 * math.pi * np.linalg.inv(lattice).T
    qmax = max(np.linalg.norm(np.array(q) @ Bn) for q in grid)
    gm = np.ceil((kc + qmax) * np.linalg.norm(lattice, axis=1) / (2 * math.pi)).astype(int) + 1
    ms = np.stack(np.meshgrid(*[np.arange(-m, m + 1) for m in gm], indexing="ij"), -1).reshape(-1, 3)
    total = {id(x): torch.zeros_like(x) for x in (R, A, *leaf)}
    E = 0.0
    for kq in grid:
        kn = np.linalg.norm((ms + np.array(kq)) @ Bn, axis=1)
        m = torch.tensor(ms[(kn < kc) & (kn > 1e-12)], **f64)
        B = 2 * math.pi * torch.linalg.inv(A).T
        q = torch.tensor(kq, **f64) @ B
        r, d = pairs()
        x = gam * d
        ex, ec = 2.0 / math.sqrt(math.pi) * x * torch.exp(-x * x), torch.erfc(x)
        lost = 1.0 - _fermi(d, rad[pi] + rad[pj], BETA, STEEP)
        P, W = (ec + ex - lost) / d ** 3, -(3 * ec + ex * (3 + 2 * x * x) - 3 * lost) / d ** 5
        T = P[:, None, None] * eye + W[:, None, None] * (r[:, :, None] * r[:, None, :])
        T = summed(T * torch.exp(-1j * (r @ q))[:, None, None])
        G = m @ B
        k = G + q
        k2 = (k * k).sum(-1)
        f = 4 * math.pi / torch.linalg.det(A).abs() * torch.exp(-k2 / (4 * gam * gam)) / k2
        S = torch.exp(1j * (R @ G.T))   # [n, G]
        T = T + torch.stack([torch.stack([(S.conj() * (f * k[:, e] * k[:, c])) @ S.T for c in range(3)], -1)
                             for e in range(3)], -2).permute(0, 2, 1, 3).reshape(3 * n, 3 * n)
        T = T - 4 * gam ** 3 / (3 * math.sqrt(math.pi)) * torch.eye(3 * n, **f64)
        c3 = (om * a.sqrt()).repeat_interleave(3)
        Q = c3[:, None] * c3[None, :] * T + torch.diag((om * om).repeat_interleave(3))
        e = 0.5 / len(grid) * torch.linalg.eigvalsh(0.5 * (Q + Q.conj().T)).sqrt().sum()
        for x, gx in zip((R, A, *leaf), torch.autograd.grad(e, (R, A, *leaf))):
            total[id(x)] += gx
        E = E + e.detach()
    E = E - 1.5 * om.detach().sum()
    total[id(om)] -= 1.5
    grads = torch.autograd.grad(scr, ins, [total[id(x)] for x in leaf], allow_unused=True)
    grads = [g if g is not None else torch.zeros_like(x) for g, x in zip(grads, ins)]
    return E, [grads[0] + total[id(R)], *grads[1:5]], a.detach(), grads[5] + total[id(A)]


def _exact_ts(coords, par):
    R, p0, p1, p2, p3 = ins = [torch.tensor(x, dtype=torch.float64, device=_device(), requires_grad=True)
                               for x in (coords, *par)]
    n = R.shape[0]
    self_ = torch.eye(n, dtype=torch.bool, device=R.device)
    a, om, rv = p0 * p3, 4.0 * p1 / (3.0 * p0 ** 2), p2 * p3 ** (1.0 / 3.0)
    r = R[None] - R[:, None]
    d = torch.where(self_, torch.ones((), dtype=R.dtype, device=R.device), (r * r).sum(-1)).sqrt()
    c6 = 1.5 * a[:, None] * a[None, :] / (1.0 / om[:, None] + 1.0 / om[None, :])
    E = -0.5 * (torch.where(self_, torch.zeros_like(d), c6 * _fermi(d, rv[:, None] + rv[None, :], S_R, 20.0) / d ** 6)).sum()
    return E.detach(), torch.autograd.grad(E, ins)


def _exact_train(case, seed):
    dev = _device()
    X, Y, p, m, v, mean, std, idx = [torch.tensor(x, device=dev) for x in _train_data(case, seed)]
    p16 = p.to(torch.float16).double().requires_grad_(True)
    F = learned.F
    cut = np.cumsum([0, F * 128, 128, 128 * 128, 128, 128 * 16, 16])
    outs, losses = [], []
    for k in range(MEMBERS):
        W1, b1, W2, b2, W3, b3 = [p16[k, i:j] for i, j in zip(cut, cut[1:])]
        x = (X[idx[k].long()].double() - mean.double()) / std.double()
        h = torch.nn.functional.silu(x @ W1.reshape(F, 128) + b1)
        h = torch.nn.functional.silu(h @ W2.reshape(128, 128) + b2)
        y = h @ W3.reshape(128, 16) + b3
        outs.append(y)
        losses.append(((y - Y[idx[k].long()].double()) ** 2).mean())
    g, = torch.autograd.grad(sum(losses), p16)
    m1 = 0.9 * m.double() + 0.1 * g
    v1 = 0.999 * v.double() + 0.001 * g * g
    step = m1 / (1 - 0.9 ** TRAIN_STEP) / (torch.sqrt(v1 / (1 - 0.999 ** TRAIN_STEP)) + 1e-8)
    return {"loss": torch.stack(losses).detach(), "outputs": torch.stack(outs).detach(), "grad": g,
            "params": p.double() - LR * step, "m": m1, "v": v1}


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case.get("scs") == "learned" or case["n"] > (1100 if "k" not in case else 100) and case["kind"] != "ts":
        return None   # the model's fitted screening has no closed form; large spectra take too long
    coords, par, lattice, k_grid = _system(case, seed)
    if case["kind"] == "ts":
        E, g = _exact_ts(coords, par)
        return {"energy": E.item(), "grad_coords": g[0].cpu().numpy(), "grad_params": torch.stack(g[1:]).cpu().numpy()}
    if lattice is not None:
        E, g, a, gA = _exact_cell(case, coords, par, lattice, k_grid)
    else:
        E, g, a = _exact_cluster(case, coords, par)
    gp = torch.stack(list(g[1:]))
    if case["kind"] == "autograd":
        return {"energy": E, "grad_coords": g[0], "grad_params": list(gp)}
    if case["kind"] == "device":
        return {"energy": E.reshape(1), "grad_coords": g[0], "alpha": a, "grad_params": gp}
    out = {"energy": E.item(), "grad_coords": g[0].cpu().numpy(), "grad_params": gp.cpu().numpy(),
           "alpha": a.cpu().numpy()}
    if lattice is not None:
        out["grad_lattice"] = gA.cpu().numpy()
    return out
