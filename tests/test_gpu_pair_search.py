"""GPU checks of the pair search at the sizes where its warps, cells and runs
can go wrong, against the oracle: one cell only, three cells a side (every run
of cells crosses the box), many cells, fewer beads than a warp, and lists that
overflow their first capacity.  The interparticle forces and the lubrication
operator see every pair of their cut-offs, so a missing or doubled pair shows.
FP64 on both sides with the same pair rule: relative 1e-12."""

import numpy as np
import pytest

import oracle as O
import synth
from oracle import contact_oracle as C

pytestmark = pytest.mark.gpu


def oracle_args(d):
    return dict(kn=d["kn"], A_H=d["hamaker"], Z=d["zeta"], kappa=d["kappa"], h_c=d["h_c"], r_cut=d["r_cut"])


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g

    g.build()
    import paper_2607_25161_gb300 as p

    return p


@pytest.mark.parametrize("n_agg,nb,L,xi", [(5, 1, 9.0, 2.0), (40, 2, 12.5, 2.0), (97, 3, 22.0, 1.6),
                                           (150, 2, 40.0, 2.0)])
@pytest.mark.parametrize("tilt", [0.0, 2.3])
def test_forces_and_lubrication_see_every_pair(pkg, n_agg, nb, L, xi, tilt):
    rng = np.random.default_rng(n_agg)
    shapes = [synth.random_attachment_aggregate(nb, rng) for _ in range(n_agg)]
    pos, body = synth.pack_suspension(shapes, L, rng, h_gen=0.05)
    dlvo = dict(kn=2.5e3, hamaker=15.0, zeta=4.0, kappa=1.0, h_c=0.03, r_cut=3.4)
    s = pkg.Suspension(pos, body, L, xi=xi, xerr=1e-6, lub_cutoff=3.0, tilt=tilt)
    got = s.interparticle(**dlvo)
    ref, _ = C.pair_forces(pos, body, L, tilt=tilt, **oracle_args(dlvo))
    assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)
    sd = O.assemble(pos, body, L, gamma=0.0, rlub=3.0, tilt=tilt, M=np.eye(11 * len(pos)))
    dU = rng.normal(size=(n_agg, 6))
    want = (sd["RRFU"] @ dU.reshape(-1)).reshape(-1, 6)
    lub = s.apply_lubrication(dU, pkg.FSD_FP64)
    s.close()
    assert np.linalg.norm(lub - want) <= 1e-12 * max(np.linalg.norm(want), 1.0)


def test_lists_grow_past_their_first_capacity(pkg):
    # a dense cluster in a large box: the capacities follow the mean density
    rng = np.random.default_rng(3)
    core, _ = synth.pack_suspension([np.zeros((1, 3))] * 300, 20.0, rng, h_gen=0.02)
    pos = core + 30.0
    L = 90.0
    body = np.arange(300)
    dlvo = dict(kn=2.5e3, hamaker=15.0, zeta=4.0, kappa=1.0, h_c=0.03, r_cut=5.0)
    s = pkg.Suspension(pos, body, L, xi=0.3, lub_cutoff=5.0)
    got = s.interparticle(**dlvo)
    s.close()
    ref, _ = C.pair_forces(pos, body, L, **oracle_args(dlvo))
    assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)
