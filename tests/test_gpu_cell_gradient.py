"""The cell gradient's sums as products (k_qgrad.cu) against the oracle: odd atom counts, k-grids with and without
Gamma, few and many images, atoms outside the cell."""
import numpy as np
import pytest

import oracle as o
from paper_2308_03140_gb300 import binding
from paper_2308_03140_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,edge,grid,gamma,shift", [(1, 6.0, (1, 1, 1), 0.5, 0.0), (7, 9.0, (2, 1, 3), 0.45, 0.0),
                                                   (17, 11.0, (1, 2, 1), 0.3, 40.0), (33, 13.0, (3, 1, 1), 0.6, -25.0)])
def test_cell_gradients_against_the_oracle(N, edge, grid, gamma, shift):
    s = syn.triclinic_cell(N, edge=(edge, 1.2 * edge), k_grid=grid, seed=N)
    R = s.coords + shift * np.array([1.0, -0.5, 0.25])
    R[N // 2] += 2.0 * s.lattice[1] - s.lattice[0]
    p = (s.alpha0_ref, s.c6_ref, s.rvdw_ref, s.ratio)
    rc, kc = 6.5 / gamma, 11.0 * gamma
    with binding.MBD(0, ewald_gamma=gamma, real_cutoff=rc, recip_cutoff=kc) as m:
        m.set_geometry(R, s.lattice, grid)
        m.set_free_atom_params(*p)
        E, gR, gp, _ = m.evaluate(True)
        gA = m.lattice_gradient()
    kap = o.monkhorst_pack(grid)
    E_ref = o.periodic_rsscs_energy(R, s.lattice, kap, *p, gamma, rc, kc)
    _, gR_ref, gA_ref, gp_ref = o.periodic_rsscs_gradient(R, s.lattice, kap, *p, gamma, rc, kc)
    # the bounds of the periodic parity test (FP64)
    assert abs(E - E_ref) <= 1e-9 * max(abs(E_ref), 1e-6)
    assert np.max(np.abs(gR - gR_ref)) <= 1e-8
    assert np.max(np.abs(gA - gA_ref)) <= 1e-8 * max(1.0, np.max(np.abs(gA_ref)))
    for k in range(4):
        assert np.max(np.abs(gp[k] - gp_ref[k])) <= 1e-8 * max(1.0, np.max(np.abs(gp_ref[k])))
