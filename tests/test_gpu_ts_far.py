"""TS pairs so far apart that their squared distance overflows contribute nothing, as at any large distance."""
import numpy as np
import pytest

from paper_2308_03140_gb300 import binding, build
from paper_2308_03140_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("far", [1e153, 1e155])
def test_far_pairs_contribute_nothing(far):
    build.build()
    s = syn.sphere_cluster(40, seed=9)
    par = (s.alpha0_ref, s.c6_ref, s.rvdw_ref, s.ratio)
    with binding.MBD(0) as m:
        m.set_geometry(s.coords)
        m.set_free_atom_params(*par)
        E, gR, gp = m.ts_energy(0.94)
        m.set_geometry(np.concatenate([s.coords, [[far, 0.0, -far]]]))
        m.set_free_atom_params(*(np.append(x, x[0]) for x in par))
        E2, gR2, gp2 = m.ts_energy(0.94)
    assert abs(E2 - E) <= 1e-14 * abs(E) and np.allclose(gR2[:40], gR, rtol=1e-13, atol=1e-18)
    assert np.all(gR2[40] == 0.0) and np.all(gp2[:, 40] == 0.0) and np.allclose(gp2[:, :40], gp, rtol=1e-13, atol=0)
