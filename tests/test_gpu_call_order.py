"""What one call leaves for the next.  fsd_contact_forces prepares the whole
geometry and the next solve keeps it; a mobility application in between
prepares the lists alone and must not take anything from that solve.

A body of two beads 6e7 radii apart has a per-aggregate block whose
translational pivot (2 zeta0) is below 1e-14 of its largest entry
(2 zeta0 (3e7)^2): singular to working precision, which the solve reports."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g

    g.build()
    import paper_2607_25161_gb300 as p

    return p


@pytest.mark.parametrize("flags", [0, 4])  # the host-driven loop and the captured one
def test_singular_block_is_reported_after_a_mobility_call(pkg, flags):
    L = 4e8
    pos = np.array([[1e8, 1e8, 1e8], [1.6e8, 1e8, 1e8]])
    s = pkg.Suspension(pos, np.zeros(2), L, xi=1.0, rc=10.0, grid=16, P=8, restart=2, max_iter=2, flags=flags)
    for mobility in (False, True):
        s.contact(1e4)
        if mobility:
            s.apply_mobility(np.ones((2, 11)))
        with pytest.raises(pkg.FsdError, match="singular"):
            s.solve(np.ones((1, 6)), 0.0)
    s.close()


def test_mobility_between_forces_and_solve_changes_nothing(pkg):
    pos, body, L = synth.suspension(40, 4, 0.1, 9)
    ft = synth.random_forces(40, 9)
    prm = dict(lub_cutoff=3.0, precision=pkg.FSD_MIXED, xi=0.9)
    s = pkg.Suspension(pos, body, L, **prm)
    want = s.solve(ft, 1.0)[:2]
    s.close()
    s = pkg.Suspension(pos, body, L, **prm)
    s.contact(1e4)
    s.apply_mobility(np.ones((160, 11)), precision=pkg.FSD_MIXED)
    got = s.solve(ft, 1.0)[:2]
    s.close()
    # the same kernels on the same lists (a second refinement sweep's FP64
    # spreading sums with atomics)
    for x, y in zip(got, want):
        assert np.linalg.norm(x - y) <= 1e-9 * np.linalg.norm(y)
