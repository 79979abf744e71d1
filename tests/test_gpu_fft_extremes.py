"""GPU parity of the wave-space operator at the ends of its grid sizes: the
smallest grids (8, 10 and 12 points a side: x tiles wider than the grid, the
smallest register DFTs, windows as wide as the box), the largest of the
two-factor passes (400 = 20 x 20) and the staged plan beside and above it
(384, a multiple of 4, and 432).

The smallest grids are too coarse for the wave-vector sum, so they are held
against the discretised operator itself (spreading, plain DFT, Green's
function, interpolation) in numpy.  Tolerances (relative L2), set before the
first run: 1e-12 in FP64 against numpy (the same sums in another order; the
window deconvolution and the Ewald filter cancel to within a factor e^2 at
these sizes), 2e-5 in FP32.  The largest: 1e-6 in FP64 at P = 16 against the
oracle's wave-vector sum, and in FP32 2e-5 n / 64, as FP32 positions move the
window weights in proportion to n."""

import ctypes

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

FP64, MIXED = 0, 1
L, XI = 8.0, 0.7


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g

    g.build()
    import paper_2607_25161_gb300 as p

    return p


def strain(s):
    r2, r6 = 0.5 ** 0.5, 6.0 ** -0.5
    xx, yy, zz = r2 * s[0] - r6 * s[1], -r2 * s[0] - r6 * s[1], 2 * r6 * s[1]
    return np.array([[xx, r2 * s[2], r2 * s[3]], [r2 * s[2], yy, r2 * s[4]], [r2 * s[3], r2 * s[4], zz]])


def five(e):
    e = 0.5 * (e + e.T)
    r2, r6 = 0.5 ** 0.5, 6.0 ** -0.5
    return np.array([r2 * (e[0, 0] - e[1, 1]), r6 * (2 * e[2, 2] - e[0, 0] - e[1, 1]), e[0, 1] / r2, e[0, 2] / r2,
                     e[1, 2] / r2])


def discrete_wave(pos, F, n, P):
    """The operator on the grid [z][y][x], a = eta = 1.  The six real fields
    travel as g_p + i g_(p+3); a grid index k <= n/2 stands for itself, one
    beyond for k - n; wave vectors with kx > n/2 follow as conjugates."""
    h = L / n
    ms = 0.976 * np.sqrt(np.pi * P)
    al = 2.0 * ms * ms / (P * h) ** 2
    cn = (al / np.pi) ** 1.5
    grid = np.zeros((6, n, n, n))
    window = []
    for p, f in zip(pos, F):
        g = np.floor(p / h).astype(int)[:, None] - P // 2 + 1 + np.arange(P)
        y = g * h - p[:, None]
        w = np.exp(-al * y * y)
        W = cn * w[2][:, None, None] * w[1][None, :, None] * w[0][None, None, :]
        Y = (y[0][None, None, :], y[1][None, :, None], y[2][:, None, None])
        ix = np.ix_(g[2] % n, g[1] % n, g[0] % n)
        lx = f[3:6]
        D = strain(f[6:]) + 0.5 * np.array([[0, -lx[2], lx[1]], [lx[2], 0, -lx[0]], [-lx[1], lx[0], 0]])
        for c in range(3):
            grid[c][ix] += W * f[c]
            grid[3 + c][ix] += 2 * al * W * sum(D[c, e] * Y[e] for e in range(3))
        window.append((ix, W, Y))
    s = np.fft.fftn(grid, axes=(1, 2, 3))
    k1 = np.arange(n)
    k1 = np.where(k1 <= n // 2, k1, k1 - n).astype(float)
    kv = np.stack(np.broadcast_arrays(k1[None, None, :], k1[None, :, None], k1[:, None, None]))
    m = (kv ** 2).sum(0)
    m[0, 0, 0] = 1.0
    k2 = m * (2 * np.pi / L) ** 2
    A = (1 + k2 / (4 * XI ** 2)) * np.exp(-k2 / (4 * XI ** 2) + k2 / (2 * al)) / k2 / n ** 3
    A[0, 0, 0] = 0.0
    z = np.sqrt(k2)
    fm, fd = np.sin(z) / z, 3 * (np.sin(z) - z * np.cos(z)) / z ** 3
    v = A * (fm * s[:3] + fd * s[3:])
    v = v - kv * (kv * v).sum(0) / m
    u = np.concatenate([fm * v, fd * v])
    # kx > n/2: the conjugates of the half spectrum's values at -k
    mirror = (-np.arange(n)) % n
    half = np.conj(u[:, mirror][:, :, mirror][:, :, :, mirror])
    u[..., n // 2 + 1:] = half[..., n // 2 + 1:]
    t = np.fft.ifftn(u[:3] + 1j * u[3:], axes=(1, 2, 3)) * n ** 3
    f = np.concatenate([t.real, t.imag])
    out = np.zeros((len(pos), 11))
    for i, (ix, W, Y) in enumerate(window):
        W = W * h ** 3
        G = np.array([[(2 * al * W * Y[e] * f[3 + c][ix]).sum() for e in range(3)] for c in range(3)])
        out[i, :3] = [(W * f[c][ix]).sum() for c in range(3)]
        out[i, 3:6] = 0.5 * np.array([G[2, 1] - G[1, 2], G[0, 2] - G[2, 0], G[1, 0] - G[0, 1]])
        out[i, 6:] = five(G)
    return out


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("n,P", [(8, 4), (8, 6), (8, 8), (10, 6), (10, 10), (12, 8), (12, 12)])
def test_wave_operator_on_the_smallest_grids(pkg, n, P):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(100 * n + P)
    pos = rng.uniform(0.0, L, size=(5, 3))
    F = rng.normal(size=(5, 11))
    ref = discrete_wave(pos, F, n, P)
    s = pkg.Suspension(pos, np.arange(5), L, xi=XI, rc=3.5, grid=n, P=P, restart=2, inner_restart=2)
    assert rel(s.apply_mobility(F, part=2, precision=FP64), ref) <= 1e-12
    assert rel(s.apply_mobility(F, part=2, precision=MIXED), ref) <= 2e-5
    s.close()
    dpos, dF = (torch.tensor(a, dtype=torch.float64, device="cuda") for a in (pos, F))
    out = torch.full((5, 11), float("nan"), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    st = pkg.load().fsd_apply_wave_noalloc(5, *(ctypes.c_void_p(t.data_ptr()) for t in (dpos, dF, out)), L, XI, n, P,
                                           0.0, 1.0, 1.0, None)
    torch.cuda.synchronize()
    assert st == pkg.FSD_OK
    assert rel(out.cpu().numpy(), ref) <= 2e-5


@pytest.mark.parametrize("n", [384, 400, 432])
def test_wave_operator_on_the_largest_grids(pkg, n):
    rng = np.random.default_rng(21)
    pos = rng.uniform(0.0, L, size=(5, 3))
    F = rng.normal(size=(5, 11))
    for tilt in (0.0, 1.7):
        M = O.mobility_wave_dense(pos, L, XI, 2 * XI * np.sqrt(46.0), tilt=tilt)
        ref = (M.reshape(55, 55) @ F.reshape(-1)).reshape(5, 11)
        s = pkg.Suspension(pos, np.arange(5), L, xi=XI, rc=3.5, grid=n, P=16, xerr=1e-8, tilt=tilt, restart=2,
                           inner_restart=2)
        assert rel(s.apply_mobility(F, part=2, precision=FP64), ref) <= 1e-6
        assert rel(s.apply_mobility(F, part=2, precision=MIXED), ref) <= 2e-5 * n / 64.0
        s.close()
