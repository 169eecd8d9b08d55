"""Q(q) of cells built with its reciprocal sums as products on the tensor cores, and the build on
the FP64 pipe that a long real-space cutoff selects (its image table would be too large), each against
the CPU oracle (oracle/mbd_periodic.c) at the same cutoffs, which also end the screening's image sums:
energies to 1e-10 relative, gradients to 1e-8, as on the periodic path."""
import pytest

from paper_2308_03140_gb300 import binding, build
from test_gpu_periodic import run_both, small_cell

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    binding.load()


def evaluate(R, A, p, grid, gamma, rc, kc):
    with binding.MBD(0, ewald_gamma=gamma, real_cutoff=rc, recip_cutoff=kc) as m:
        m.set_geometry(R, A, grid)
        m.set_free_atom_params(*p)
        return m.evaluate(True)[0]


# one atom; ragged 16-atom tiles; rows of the operands just over a 256-row tile (6 N = 258); odd grids
@pytest.mark.parametrize("N,edge,grid", [(1, 5.0, (3, 2, 1)), (2, 6.0, (2, 2, 2)), (17, 11.0, (1, 1, 2)),
                                         (43, 15.0, (1, 1, 1))])
def test_both_builds_against_the_oracle(N, edge, grid):
    R, A, p = small_cell(N, edge, 40 + N)
    gamma, kc = 0.3, 11 * 0.3
    run_both(R, A, p, grid, gamma, 6.5 / gamma, kc)
    run_both(R, A, p, grid, gamma, 7.0 * edge, kc)   # over 14^3 image offsets


def test_one_context_through_both_builds():
    # the lattice alone decides: the second geometry keeps atoms and grid in a smaller cell (2184 image
    # offsets, 1210 before), the third goes back; each agrees with a fresh context
    R, A, p = small_cell(2, 9.0, 51)
    gamma, rc, kc = 0.5, 45.0, 5.5
    with binding.MBD(0, ewald_gamma=gamma, real_cutoff=rc, recip_cutoff=kc) as m:
        for f in (1.0, 0.8, 1.0):
            m.set_geometry(f * R, f * A, (1, 1, 1))
            m.set_free_atom_params(*p)
            E = m.evaluate(True)[0]
            Ef = evaluate(f * R, f * A, p, (1, 1, 1), gamma, rc, kc)
            assert abs(E - Ef) <= 1e-12 * abs(Ef)


def test_oracle_at_one_atom():
    R, A, p = small_cell(1, 6.0, 61)
    run_both(R, A, p, (2, 1, 2), 0.35, 6.5 / 0.35, 11 * 0.35)
