"""The FP64 SCS adjoint pass over tiles of 32 x 32 atoms: sizes around a tile's edge, and its three groupings of the
frequencies (one, two and four a CTA), against the oracle's gradients."""
import numpy as np
import pytest

import oracle as o
from paper_2308_03140_gb300 import binding
from paper_2308_03140_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,n_freq", [(1, 15), (31, 15), (33, 15), (64, 15), (33, 19), (197, 15)])
def test_gradients_against_the_oracle(N, n_freq):
    s = syn.cube_cluster(N, 14.0 * (max(N, 8) / 32.0) ** (1.0 / 3.0), 2.5, seed=N)
    with binding.MBD(0, n_freq=n_freq) as m:
        m.set_geometry(s.coords)
        m.set_free_atom_params(s.alpha0_ref, s.c6_ref, s.rvdw_ref, s.ratio)
        E, gR, gp, _ = m.evaluate(True)
    E_ref, gR_ref, gp_ref = o.mbd_rsscs_gradient(*o.system_args(s), n_freq=n_freq, mode="adjoint")
    # the bounds of the small clusters' parity test: FP64 through Newton-Schulz
    assert abs(E - E_ref) <= 1e-9 * max(abs(E_ref), 1e-6)
    assert np.max(np.abs(gR - gR_ref)) <= 1e-8
    for k in range(4):
        assert np.max(np.abs(gp[k] - gp_ref[k])) <= 1e-8 * max(1.0, np.max(np.abs(gp_ref[k])))
