"""The no-allocation wave-space entry point at bead counts around its blocks of
32 beads, and on grids whose twiddles fill one block of 32 or spill into a
second and whose fields are planar (30) or bricked.  Checked against the
context's wave-space operator (fsd_apply_mobility, part 2, FP32) within the
FP32 operator tolerance of the parity tests, 2e-5 relative L2."""

import ctypes

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_beads,grid", [(1, 30), (31, 32), (32, 30), (33, 36), (97, 48)])
def test_noalloc_wave_at_block_edges(n_beads, grid):
    torch = pytest.importorskip("torch")
    import __graft_entry__ as g

    g.build()
    import paper_2607_25161_gb300 as pkg

    lib = pkg.load()
    xi, P = 0.6, 8
    phi = n_beads * 4.0 / 3.0 * np.pi / 17.3**3  # R_c = 8.2 < L / 2; 30 points resolve xi
    pos, body, L = synth.suspension(n_beads, 1, phi, 41)
    s = pkg.Suspension(pos, body, L, xi=xi, grid=grid, P=P)
    F = np.random.default_rng(42).normal(size=(n_beads, 11))
    ref = np.asarray(s.apply_mobility(F, part=2, precision=pkg.FSD_MIXED))
    s.close()
    dpos = torch.tensor(pos, dtype=torch.float64, device="cuda")
    dF = torch.tensor(F, dtype=torch.float64, device="cuda")
    dout = torch.full((n_beads, 11), float("nan"), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    st = lib.fsd_apply_wave_noalloc(n_beads, ctypes.c_void_p(dpos.data_ptr()), ctypes.c_void_p(dF.data_ptr()),
                                    ctypes.c_void_p(dout.data_ptr()), L, xi, grid, P, 0.0, 1.0, 1.0, None)
    torch.cuda.synchronize()
    assert st == pkg.FSD_OK
    got = dout.cpu().numpy()
    assert np.all(np.isfinite(got))
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) < 2e-5
