"""Mixed-precision cells iterate on several Bloch vectors at a time (mixed_group in mbd_api.cu): a grid of more
vectors than a group holds (16 + 2), and the forms of the GEMM that take a group's matrices one by one, against
the FP64 path of the same cell."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2308_03140_gb300 import binding
from paper_2308_03140_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu
# energy per atom and largest relative gradient error of the mixed modes on cells (test_gpu_periodic.py)
BOUNDS = {"tf32x3": (5e-8, 2e-4), "bf16x3": (1e-7, 1e-3)}
PREC = {"fp64": binding.MBD_PREC_FP64, "tf32x3": binding.MBD_PREC_TF32X3, "bf16x3": binding.MBD_PREC_BF16X3}
N, GRID = 23, (3, 3, 2)


def evaluate(precision):
    s = syn.triclinic_cell(N, edge=(9.0, 11.5), k_grid=GRID, seed=5)
    with binding.MBD(0, precision=PREC[precision], ewald_gamma=0.3, real_cutoff=6.5 / 0.3, recip_cutoff=3.3) as m:
        m.set_geometry(s.coords, s.lattice, GRID)
        m.set_free_atom_params(s.alpha0_ref, s.c6_ref, s.rvdw_ref, s.ratio)
        E, gR, gp, _ = m.evaluate(True)
        return np.concatenate([[E], gR.ravel(), m.lattice_gradient().ravel(), gp.ravel()])


def check(x, ref, precision):
    e, g = BOUNDS[precision]
    assert abs(x[0] - ref[0]) <= e * N, (x[0], ref[0])
    for a, b in [(1, 1 + 3 * N), (1 + 3 * N, 10 + 3 * N)] + [(10 + 3 * N + k * N, 10 + 3 * N + (k + 1) * N) for k in range(4)]:
        assert np.abs(x[a:b] - ref[a:b]).max() <= g * np.abs(ref[a:b]).max()


@pytest.mark.parametrize("precision", ["tf32x3", "bf16x3"])
def test_more_bloch_vectors_than_a_group(precision):
    check(evaluate(precision), evaluate("fp64"), precision)


@pytest.mark.parametrize("form", ["single", "pair"])
def test_other_forms_take_a_group_one_by_one(form, tmp_path):
    out = tmp_path / "x.npy"
    code = f"import numpy as np, test_gpu_cell_groups as t; np.save({str(out)!r}, t.evaluate('bf16x3'))"
    here = os.path.dirname(os.path.abspath(__file__))
    env = dict(os.environ, MBDGB_TC_FORM=form, PYTHONPATH=os.pathsep.join([here, os.path.dirname(here)]))
    subprocess.run([sys.executable, "-c", code], env=env, check=True, timeout=300)
    check(np.load(out), evaluate("fp64"), "bf16x3")
