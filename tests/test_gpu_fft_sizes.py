"""GPU parity of the wave-space operator over the FFT sizes: every way the
transform is split (two register DFTs of each radix from 3 to 20, and the
staged plan of the sizes without a two-factor kernel), with tiles that divide
the grid and tiles that do not, in the cube and in the sheared box, against
the oracle's wave-vector sum.

Tolerances (relative L2), set before the first run: 1e-6 in FP64 at P = 16
(the window error is about 1e-8 there).  FP32 positions are rounded to about
6e-8 L, which moves a window weight by about 1.5 x 6e-8 L / h = 9e-8 n
relative: 2e-5, as for the FP32 operator elsewhere, up to n = 64 and in
proportion to n beyond."""

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

FP64, MIXED = 0, 1
L, XI = 8.0, 0.7
SIZES = [16, 18, 20, 24, 30, 32, 36, 40, 48, 50, 54, 60, 64, 72, 80, 90, 96, 100, 108, 120, 128, 144, 150,
         160, 162, 180, 192, 200, 216, 240, 250, 256, 270, 288, 300, 320, 324, 360]


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g

    g.build()
    import paper_2607_25161_gb300 as p

    return p


@pytest.fixture(scope="module")
def refs():
    rng = np.random.default_rng(21)
    pos = rng.uniform(0.0, L, size=(5, 3))
    F = rng.normal(size=(5, 11))
    kmax = 2 * XI * np.sqrt(46.0)
    out = {}
    for tilt in (0.0, 1.7):
        M = O.mobility_wave_dense(pos, L, XI, kmax, tilt=tilt)
        out[tilt] = (M.reshape(55, 55) @ F.reshape(-1)).reshape(5, 11)
    return pos, F, out


@pytest.mark.parametrize("n", SIZES)
def test_wave_operator_over_grid_sizes(pkg, refs, n):
    pos, F, out = refs
    for tilt, ref in out.items():
        s = pkg.Suspension(pos, np.arange(5), L, xi=XI, rc=3.5, grid=n, P=16, xerr=1e-8, tilt=tilt,
                           restart=2, inner_restart=2)
        for prec, tol in ((FP64, 1e-6), (MIXED, 2e-5 * max(1.0, n / 64.0))):
            got = s.apply_mobility(F, part=2, precision=prec)
            assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref), (n, tilt, prec)
        s.close()


@pytest.mark.parametrize("n", [18, 30, 64, 108, 250])
def test_brownian_wave_field_over_grid_sizes(pkg, refs, n):
    # the same counter-based field in both precisions (psi_real = 0 leaves the
    # wave part alone): the samples agree as the two operators do
    pos, _, _ = refs
    res = {}
    for prec in (FP64, MIXED):
        s = pkg.Suspension(pos, np.arange(5), L, xi=XI, rc=3.5, grid=n, P=16, xerr=1e-8, precision=prec,
                           restart=2, inner_restart=2, lanczos_max_iter=2)
        zero = np.zeros((5, 11))
        slip, _, _ = s.brownian(1.0, 1e-3, seed=3, step=1, psi_real=zero)
        res[prec] = slip
        s.close()
    assert np.abs(res[FP64]).max() > 0
    tol = 2e-5 * max(1.0, n / 64.0)
    assert np.linalg.norm(res[MIXED] - res[FP64]) <= tol * np.linalg.norm(res[FP64])
