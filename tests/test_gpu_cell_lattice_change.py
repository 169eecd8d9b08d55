"""A lattice that changes between evaluations by so little that the context's lists keep their sizes, but with more image
offsets inside the real-space cutoff: parameters and workspace stay, as for any other change of coordinates."""
import numpy as np
import pytest

from paper_2308_03140_gb300 import binding, build
from paper_2308_03140_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu
RC = 40.0


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    binding.load()


def cell(n=24):
    s = syn.sphere_cluster(n, seed=77)
    lo = s.coords.min(0)
    return s, s.coords - lo, np.ptp(s.coords, axis=0)


@pytest.mark.parametrize("precision", ["MBD_PREC_FP64", "MBD_PREC_BF16X3"])
def test_parameters_stay_when_the_image_tables_grow(precision):
    s, R, size = cell()
    # 2 RC / a just below an integer m, then just above it: m + 1 offsets in each direction, then m + 2
    m = int(np.floor(2.0 * RC / (size.max() + 4.0)))
    assert m >= 1
    small, large = np.eye(3) * (2.0 * RC / m) * (1.0 + 1e-6), np.eye(3) * (2.0 * RC / m) * (1.0 - 1e-6)
    opts = dict(precision=getattr(binding, precision), ewald_gamma=0.15, real_cutoff=RC, recip_cutoff=0.837)
    par = (s.alpha0_ref, s.c6_ref, s.rvdw_ref, s.ratio)
    out = {}
    with binding.MBD(0, **opts) as calc:
        calc.set_geometry(R, small, (1, 1, 2))
        calc.set_free_atom_params(*par)
        calc.evaluate(True)
        for name, lat in (("large", large), ("small", small), ("large again", large)):
            calc.set_geometry(R, lat, (1, 1, 2))
            out[name] = (*calc.evaluate(True), calc.lattice_gradient())   # the parameters of before
    for name, lat in (("large", large), ("small", small), ("large again", large)):
        with binding.MBD(0, **opts) as calc:
            calc.set_geometry(R, lat, (1, 1, 2))
            calc.set_free_atom_params(*par)
            fresh = (*calc.evaluate(True), calc.lattice_gradient())
        for x, y in zip(out[name], fresh):
            x, y = np.asarray(x), np.asarray(y)
            assert np.abs(x - y).max() <= 1e-12 * np.abs(y).max(), name   # (sums by FP64 atomics)
