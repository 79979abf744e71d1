"""Interparticle forces with a cut-off at the edge of what the box allows: two
beads whose separation along one axis is 4e-10 below half the box, within a
cut-off 1e-10 below it.  FP32 positions cannot tell which image is the nearer;
the forces take the FP64 image.  FP64 on both sides with the same pair rule:
relative 1e-12 (the force is a smooth function of the separation there)."""

import numpy as np
import pytest

from oracle import contact_oracle as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_forces_take_the_fp64_image_at_half_the_box(axis):
    import __graft_entry__ as g

    g.build()
    import paper_2607_25161_gb300 as pkg

    L = 20.0
    rc = 0.5 * L - 1e-10
    rng = np.random.default_rng(17 + axis)
    for _ in range(12):
        pos = np.tile(rng.uniform(0.0, L, size=3), (2, 1))
        pos[1, axis] = (pos[0, axis] + 0.5 * L - 4e-10) % L
        s = pkg.Suspension(pos, np.arange(2), L, xi=2.0, rc=rc, restart=2, inner_restart=2)
        got = s.interparticle(zeta=4.0, kappa=0.1, h_c=0.03, r_cut=rc)
        s.close()
        ref, _ = C.pair_forces(pos, np.arange(2), L, kn=0.0, A_H=0.0, Z=4.0, kappa=0.1, h_c=0.03, r_cut=rc)
        assert np.abs(ref[:, axis]).min() > 1e-3
        assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)
