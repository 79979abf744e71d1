"""Performance cases of the rigid-aggregate FSD library: the calls a simulation
makes, over the sizes, precisions and options it uses, and plain 64-bit torch
values of what they return.

A case is a suspension (aggregate shapes, bead volume fraction, sizes) and one
call on it.  Suspensions are packed here on the GPU: aggregates at random
centres and orientations are pushed apart until no two beads of different
bodies are closer than 2.1 radii; large ones are periodic replicas of a packed
tile (each aggregate still has its own force and torque).

The C ABI's arrays are double in every precision.  Results of the FP32
operator and of the mixed solve are taken as float32, the type whose precision
they carry, as a program that keeps them in single precision does; results of
the FP64 paths and updated positions stay double."""

import math
import os

import numpy as np
import torch

# The batched form runs one stream per system; the library's header asks for
# 32 hardware work queues, set before the CUDA context exists.
os.environ.setdefault("CUDA_DEVICE_MAX_CONNECTIONS", "32")

import paper_2607_25161_gb300 as fsd  # noqa: E402

ACCEPT = (fsd.FSD_OK, fsd.FSD_EOVERLAP)


# ------------------------------------------------------------------ cases
def listed():
    """The cases, smallest first; `iters` is the GMRES iteration count seen at
    the case's tolerance (it enters work() only)."""
    return [
        # a caller that may not allocate applies the wave-space operator to a
        # small cluster, e.g. inside its own captured loop: launches and latency
        {"name": "wave_noalloc_700", "call": "wave", "beads": 700, "grid": 40, "P": 8, "xi": 0.5, "phi": 0.1},
        # the smallest simulation: 16 touching doublets, one dilute FP64 solve
        # with the host-driven loop (the library's default flags)
        {"name": "doublets_fp64_32", "call": "solve", "shape": "aggregate", "agg": 16, "n_b": 2, "reps": 1,
         "phi": 0.0021, "precision": "fp64", "graph": False, "lub": 0.0, "xi": 0.5, "grid": 32, "P": 8, "iters": 11},
        # interparticle (Hertz and DLVO) forces of a dense suspension, once per step
        {"name": "forces_32768", "call": "forces", "shape": "aggregate", "agg": 64, "n_b": 8, "reps": 4, "phi": 0.2,
         "precision": "mixed", "lub": 3.0, "xi": 0.5},
        # FP64 mobility for a user's own solver, a tight accuracy target and a
        # user-chosen grid (not a multiple of 4), aggregates of 1 to 6 beads
        {"name": "mobility_fp64_ragged", "call": "mobility", "shape": "ragged", "agg": 500, "n_b": 6, "reps": 1,
         "phi": 0.12, "precision": "fp64", "lub": 3.0, "xi": 0.6, "xerr": 1e-8, "grid": 90, "P": 16},
        # FP32 saddle-point operator for a user's own Krylov loop, ragged bodies
        {"name": "saddle_fp32_ragged", "call": "saddle", "shape": "ragged", "agg": 281, "n_b": 9, "reps": 2,
         "phi": 0.15, "precision": "mixed", "lub": 3.0, "xi": 0.5},
        # Brownian rods with Hertz contact, one time step: the random terms, the
        # contact forces and the step (the scaling study's workload)
        {"name": "brownian_rods_8000", "call": "brownian", "shape": "rod", "agg": 125, "n_b": 8, "reps": 2,
         "phi": 0.1, "precision": "mixed", "graph": True, "lub": 3.0, "xi": 0.5, "iters": 42},
        # dilute rods with the size-dependent splitting xi = 25 / L and the FP32
        # Krylov basis: long real-space lists, a small grid
        {"name": "dilute_rods_krylov32", "call": "solve", "shape": "rod", "agg": 128, "n_b": 8, "reps": 2,
         "phi": 0.01, "precision": "mixed", "graph": True, "krylov32": True, "lub": 3.0, "xi": "25/L", "iters": 30},
        # an ensemble of small systems solved together
        {"name": "batch_12_systems", "call": "batch", "shape": "aggregate", "systems": 12, "lo": 256, "hi": 4096,
         "n_b": 6, "phi": 0.12, "precision": "mixed", "lub": 3.0, "xi": 0.5, "iters": 47},
        # the scaling study's FP64 reference solve
        {"name": "solve_fp64_4096", "call": "solve", "shape": "aggregate", "agg": 64, "n_b": 8, "reps": 2,
         "phi": 0.1, "precision": "fp64", "graph": True, "lub": 3.0, "xi": 0.5, "iters": 49},
        # the benchmark's step: 4096 8-bead aggregates in the sheared box
        {"name": "step_mixed_32768", "call": "step", "shape": "aggregate", "agg": 64, "n_b": 8, "reps": 4,
         "phi": 0.2, "precision": "mixed", "graph": True, "lub": 3.0, "rp": 2.0, "xi": 0.5, "iters": 60},
        # the size ladder's large end: grids too wide for one block's plane
        {"name": "solve_mixed_128000", "call": "solve", "shape": "aggregate", "agg": 250, "n_b": 8, "reps": 4,
         "phi": 0.2, "precision": "mixed", "graph": True, "lub": 3.0, "rp": 2.0, "xi": 0.5, "iters": 60},
    ]


def draw(rng):
    """A case of the listed ranges: another call, size, shape, fraction, type."""
    call = rng.choice(["wave", "solve", "solve", "step", "mobility", "saddle", "forces", "brownian", "batch"])

    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if call == "wave":
        grid = rng.choice([18, 20, 24, 30, 32, 36, 40, 45 + 3, 48])
        return {"call": "wave", "beads": logint(64, 4096), "grid": grid, "P": rng.choice([4, 6, 8, 10, 12, 16]),
                "xi": round(rng.uniform(0.3, 0.8), 3), "phi": round(rng.uniform(0.02, 0.2), 3)}
    shape = "rod" if call == "brownian" else rng.choice(["aggregate", "ragged", "rod"])
    n_b = 8 if shape == "rod" else rng.randint(2, 10)
    case = {"call": call, "shape": shape, "n_b": n_b, "lub": 3.0, "xi": 0.5,
            "phi": round(rng.uniform(0.02, 0.1 if shape == "rod" else 0.2), 3)}
    if call == "batch":
        return dict(case, systems=rng.randint(4, 16), lo=200, hi=logint(400, 4096), precision="mixed", iters=45)
    fp64 = call in ("solve", "step", "mobility") and rng.random() < 0.4
    total = logint(300, 6000) if fp64 else logint(300, 80000)
    mean = 0.5 * (n_b + 1) if shape == "ragged" else n_b
    reps = 1
    while total / reps ** 3 > 1600:
        reps += 1
    case.update(agg=max(8, int(round(total / reps ** 3 / mean))), reps=reps, precision="fp64" if fp64 else "mixed")
    if call in ("solve", "step", "brownian"):
        case.update(graph=rng.random() < 0.8, rp=rng.choice([2.0, 2.1]), iters=50)
        if call == "solve" and not fp64:
            case["krylov32"] = rng.random() < 0.3
            if case["phi"] < 0.06 and rng.random() < 0.5:
                case["xi"] = "25/L"
    return case


# ------------------------------------------------------------- suspensions
def _shape(kind, n_b, rng):
    """Bead offsets of one aggregate about its centroid (radius 1): a straight
    rod, or a random attachment of touching beads."""
    if kind == "rod":
        x = (np.arange(n_b) - 0.5 * (n_b - 1)) * 2.0
        return np.stack([x, np.zeros(n_b), np.zeros(n_b)], axis=1)
    pts = np.zeros((1, 3))
    while len(pts) < n_b:
        d = rng.normal(size=3)
        cand = pts[rng.integers(len(pts))] + 2.0 * d / np.linalg.norm(d)
        if np.all(((pts - cand) ** 2).sum(1) >= 4.0 * (1.0 - 1e-12)):
            pts = np.concatenate([pts, cand[None]])
    return pts - pts.mean(axis=0)


def _pack(kind, n_agg, n_b, phi, seed, reps):
    """One packed tile: positions (N, 3) and aggregate ids (N,) on the GPU, and
    its side L.  Random centres and orientations in a box of a quarter of the
    fraction, then a soft repulsion between beads of different bodies in
    turns with a compression of the centres by 2 % (half of it again where it
    stalls; a packing that jams keeps the box it reached)."""
    rng = np.random.default_rng(seed)
    # the sizes belong to the case, not to its inputs: 1, 2, .. n_b in turn
    sizes = 1 + np.arange(n_agg) % n_b if kind == "ragged" else np.full(n_agg, n_b)
    shapes = [_shape(kind, int(s), rng) for s in sizes]
    extent = 2.0 + max(float(np.linalg.norm(s[:, None] - s[None], axis=2).max()) for s in shapes)
    # a body must not meet its own image, and alone in its box fits half of it
    want = max((int(sizes.sum()) * 4.0 / 3.0 * math.pi / phi) ** (1.0 / 3.0), 2.0 * extent if reps == 1 else extent + 0.2)
    dev = "cuda"
    body = torch.from_numpy(np.repeat(np.arange(n_agg), sizes)).to(dev)
    q = rng.normal(size=(n_agg, 4))
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    w, x, y, z = q.T
    R = np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                  2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                  2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], axis=1).reshape(-1, 3, 3)
    off = torch.from_numpy(np.concatenate([s @ r.T for s, r in zip(shapes, R)])).to(dev)
    L = want * 1.6
    C = torch.from_numpy(rng.uniform(0.0, L, size=(n_agg, 3))).to(dev)
    nb = torch.from_numpy(sizes.astype(np.float64)).to(dev)[:, None]
    inertia = torch.zeros(n_agg, 1, dtype=torch.float64, device=dev).index_add_(0, body, (off * off).sum(1, True))
    same = (body[:, None] == body[None, :]).float() * 100.0
    shrink, good, done = 0.98, None, 0
    while True:
        free = False
        for it in range(180):
            done += 1
            p = (C[body] + off).float()
            d = p[None, :, :] - p[:, None, :]
            d -= L * torch.round(d / L)
            r = d.square().sum(2).sqrt_() + same
            if it % 6 == 5 and bool((r > 2.1).all()):
                free = True
                break
            f = (2.125 - r).clamp_(min=0.0) / r.clamp(min=1e-3)
            g = -(f[:, :, None] * d).sum(1).double()
            F = torch.zeros(n_agg, 3, dtype=torch.float64, device=dev).index_add_(0, body, g)
            T = torch.zeros(n_agg, 3, dtype=torch.float64, device=dev).index_add_(0, body, torch.linalg.cross(off, g))
            C = (C + 0.5 * F / nb.sqrt()) % L
            wv = (0.5 * T / (inertia + 1.0))[body]
            th = wv.norm(dim=1, keepdim=True)
            k = wv / th.clamp(min=1e-30)
            off = off * th.cos() + torch.linalg.cross(k, off) * th.sin() + k * (k * off).sum(1, True) * (1.0 - th.cos())
        if not free and good is not None:
            C, off, L = good
            shrink = 0.5 * (1.0 + shrink)
        elif not free:
            # bodies caught in one another at the loose start go elsewhere
            caught = torch.unique(body[(r <= 2.1).any(1)])
            C[caught] = torch.from_numpy(rng.uniform(0.0, L, size=(len(caught), 3))).to(dev)
            continue
        good = (C, off, L)
        if L <= want * (1 + 1e-9) or shrink > 0.996 or done > 2000:
            return C[body] + off, body, L
        Ln = max(L * shrink, want)
        C, L = C * (Ln / L), Ln


def _suspension(kind, n_agg, n_b, phi, reps, seed):
    pos, body, L = _pack(kind, n_agg, n_b, phi, seed, reps)
    shift = torch.stack(torch.meshgrid(*[torch.arange(reps, device=pos.device)] * 3, indexing="ij"), -1).reshape(-1, 3)
    pos = (pos[None] + L * shift[:, None, :]).reshape(-1, 3).contiguous()
    body = (body[None] + n_agg * torch.arange(reps ** 3, device=pos.device)[:, None]).reshape(-1)
    return pos, body.to(torch.int32).contiguous(), L * reps


def _params(case, L):
    flags = fsd.FSD_FLAG_GRAPH if case.get("graph") else 0
    if case.get("krylov32"):
        flags |= fsd.FSD_FLAG_FP32_KRYLOV
    if case["call"] == "step":
        flags |= fsd.FSD_FLAG_LEES_EDWARDS
    p = {"precision": fsd.FSD_MIXED if case["precision"] == "mixed" else fsd.FSD_FP64, "flags": flags,
         "lub_cutoff": case["lub"], "precond_cutoff": case.get("rp", 2.1)}
    xi = 25.0 / L if case["xi"] == "25/L" else case["xi"]
    # boxes too small for the cut-off of this splitting take the library's rule
    if 2.0 + math.sqrt(-math.log(case.get("xerr", 1e-6))) / xi < 0.44 * L:
        p["xi"] = xi
    elif case["call"] == "step":
        p["xi"] = 1.02 * math.sqrt(-math.log(case.get("xerr", 1e-6))) / (0.447 * L - 2.0)
    for k in ("grid", "P", "xerr"):
        if k in case:
            p[k] = case[k]
    return p


def _forces(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + 7919)
    return torch.randn(n, 6, generator=g, device="cuda", dtype=torch.float64)


def prepare(case, seed):
    if case["call"] == "wave":
        g = torch.Generator(device="cuda").manual_seed(seed)
        n = case["beads"]
        L = (n * 4.0 / 3.0 * math.pi / case["phi"]) ** (1.0 / 3.0)
        pos = L * torch.rand(n, 3, generator=g, device="cuda", dtype=torch.float64)
        x = torch.randn(n, 11, generator=g, device="cuda", dtype=torch.float64)
        return {"case": case, "L": L, "pos": pos, "x": x, "out": torch.empty_like(x), "lib": fsd.load()}
    if case["call"] == "batch":
        rng = np.random.default_rng(seed)
        systems, plist = [], []
        for k in range(case["systems"]):
            total = case["lo"] * (case["hi"] / case["lo"]) ** (k / max(1, case["systems"] - 1))
            reps = 1 if total < 1600 else 2
            mean = 0.5 * (case["n_b"] + 1) if case["shape"] == "ragged" else case["n_b"]
            pos, body, L = _suspension(case["shape"], max(4, int(total / mean / reps ** 3)), case["n_b"],
                                       case["phi"] * rng.uniform(0.5, 1.0), reps, seed * 100 + k)
            systems.append((pos.cpu().numpy(), body.cpu().numpy(), L))
            plist.append(_params(dict(case, call="solve"), L))
        b = fsd.Batch(systems, plist)
        return {"case": case, "batch": b, "ft": _forces(b.n_agg, seed).cpu().numpy()}
    pos, body, L = _suspension(case["shape"], case["agg"], case["n_b"], case["phi"], case["reps"], seed)
    if case["call"] == "forces":
        # closer bodies than the packing leaves, so that contacts and van der
        # Waals pairs exist: a rigid shift of every third aggregate
        pos = pos + 0.15 * ((body % 3) == 0).double()[:, None]
    s = fsd.Suspension(pos, body, L, **_params(case, L))
    st = {"case": case, "s": s, "pos": pos, "body": body, "L": L, "ft": _forces(s.n_agg, seed), "k": 0, "seed": seed}
    g = torch.Generator(device="cuda").manual_seed(seed)
    if case["call"] in ("mobility", "saddle"):
        n = 11 * s.n_beads + (6 * s.n_agg if case["call"] == "saddle" else 0)
        st["x"] = torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
        st["out"] = torch.empty_like(st["x"])
    st["vel"] = torch.empty(s.n_agg, 6, device="cuda", dtype=torch.float64)
    st["str"] = torch.empty(s.n_agg, 3, 3, device="cuda", dtype=torch.float64)
    torch.cuda.synchronize()  # the context works on a stream of its own
    return st


def _kept(case, *tensors):
    return [t.float() if case.get("precision", "mixed") == "mixed" else t for t in tensors]


def run(state):
    case, call = state["case"], state["case"]["call"]
    if call == "wave":
        st = state["lib"].fsd_apply_wave_noalloc(
            case["beads"], state["pos"].data_ptr(), state["x"].data_ptr(), state["out"].data_ptr(), state["L"],
            case["xi"], case["grid"], case["P"], 0.0, 1.0, 1.0, torch.cuda.current_stream().cuda_stream or None)
        if st != fsd.FSD_OK:
            raise fsd.FsdError(st, "fsd_apply_wave_noalloc")
        return _kept(case, state["out"])
    if call == "batch":
        vel, stress, _, _ = state["batch"].solve(state["ft"], 1.0, allow=ACCEPT)
        return [vel.astype(np.float32), stress.astype(np.float32)]
    s = state["s"]
    prec = fsd.FSD_MIXED if case["precision"] == "mixed" else fsd.FSD_FP64
    if call == "mobility":
        return _kept(case, s.apply_mobility(state["x"], precision=prec, out=state["out"]))
    if call == "saddle":
        return _kept(case, s.apply_saddle(state["x"], precision=prec, out=state["out"]))
    if call == "forces":
        return [s.interparticle(kn=2.5e3, hamaker=15.0, zeta=4.0, kappa=1.0, h_c=0.03, r_cut=5.0, out=state["vel"])]
    if call == "solve":
        vel, stress, _, _ = s.solve(state["ft"], 1.0, vel=state["vel"], stresslet=state["str"], allow=ACCEPT)
        return _kept(case, vel, stress)
    state["k"] += 1
    if call == "step":
        s.step(state["ft"], 1.0, 1e-3, vel=state["vel"], allow=ACCEPT)
    else:
        s.brownian(1.0, 1e-3, seed=state["seed"], step=state["k"], outputs=False)
        s.contact(1e4, out=state["ft"])
        s.step(state["ft"], 0.0, 1e-3, vel=state["vel"], allow=ACCEPT)
    pos, quat = s.beads()
    return _kept(case, state["vel"]) + [pos, quat]


# -------------------------------------------------------------------- work
def _operator_flops(case, beads, L):
    """One application of the mobility: directed pairs within R_c (350 flops
    each), spreading and interpolation over the P^3 window (18 and 24 flops a
    point), six forward and six inverse real FFTs and the Green's function."""
    lnx = math.sqrt(-math.log(case.get("xerr", 1e-6)))
    xi = 25.0 / L if case["xi"] == "25/L" else case["xi"]
    n = case.get("grid") or (2.0 * lnx * xi + 1.0) * L / math.pi
    P = case.get("P", 12)
    rc = min(2.0 + lnx / xi, 0.5 * L)
    pairs = 0.0 if case["call"] == "wave" else beads * (beads / L ** 3) * 4.0 / 3.0 * math.pi * rc ** 3
    return 350.0 * pairs + 42.0 * beads * P ** 3 + 12 * 2.5 * n ** 3 * 3.0 * math.log2(n) + 60.0 * n ** 3


def _work1(case, beads, bodies, L):
    b = beads * 24.0  # positions in
    if case["call"] == "forces":
        # search, pair forces and the aggregate sums over the pairs in reach
        return {"bytes": b + bodies * 48.0, "flops": beads * (beads / L ** 3) * 4.0 / 3.0 * math.pi * 5.0 ** 3 * 40.0}
    if case["call"] in ("wave", "mobility", "saddle"):
        extra = bodies * 96.0 if case["call"] == "saddle" else 0.0
        return {"bytes": b + beads * 176.0 + extra, "flops": _operator_flops(case, beads, L)}
    # forces in, velocities and stresslets (or positions and quaternions) out,
    # one operator application per iteration
    return {"bytes": b + bodies * (48.0 + 120.0) + beads * 24.0, "flops": case["iters"] * _operator_flops(case, beads, L)}


def work(case):
    def box(n):
        return (n * 4.0 / 3.0 * math.pi / case["phi"]) ** (1.0 / 3.0)

    if case["call"] == "wave":
        return _work1(case, case["beads"], 0, box(case["beads"]))
    if case["call"] == "batch":
        tot = {"bytes": 0.0, "flops": 0.0}
        for k in range(case["systems"]):
            n = case["lo"] * (case["hi"] / case["lo"]) ** (k / max(1, case["systems"] - 1))
            w = _work1(case, n, n / case["n_b"], box(n))
            tot = {q: tot[q] + w[q] for q in tot}
        return tot
    bodies = case["agg"] * case["reps"] ** 3
    beads = bodies * (0.5 * (case["n_b"] + 1) if case["shape"] == "ragged" else case["n_b"])
    return _work1(case, beads, bodies, box(beads))


# ------------------------------------------------------- plain 64-bit values
# The discretised positively split Ewald mobility (the same window, grid and
# cut-off as the call's parameters), the lubrication pair model and the rigid
# constraint, written with torch operations.
def _strain(s):
    """Five orthonormal coordinates -> symmetric traceless matrices."""
    r2, r6 = 0.5 ** 0.5, 6.0 ** -0.5
    xx, yy, zz = r2 * s[:, 0] - r6 * s[:, 1], -r2 * s[:, 0] - r6 * s[:, 1], 2 * r6 * s[:, 1]
    xy, xz, yz = r2 * s[:, 2], r2 * s[:, 3], r2 * s[:, 4]
    return torch.stack([xx, xy, xz, xy, yy, yz, xz, yz, zz], 1).reshape(-1, 3, 3)


def _five(e):
    """The five coordinates of the symmetric traceless part."""
    e = 0.5 * (e + e.transpose(1, 2))
    r2, r6 = 0.5 ** 0.5, 6.0 ** -0.5
    return torch.stack([r2 * (e[:, 0, 0] - e[:, 1, 1]), r6 * (2 * e[:, 2, 2] - e[:, 0, 0] - e[:, 1, 1]),
                        e[:, 0, 1] / r2, e[:, 0, 2] / r2, e[:, 1, 2] / r2], 1)


def _cross_matrix(v):
    o = torch.zeros_like(v[:, 0])
    return torch.stack([o, -v[:, 2], v[:, 1], v[:, 2], o, -v[:, 0], -v[:, 1], v[:, 0], o], 1).reshape(-1, 3, 3)


class _Mobility:
    def __init__(self, pos, L, p, real=True):
        self.pos, self.L, self.n, self.P = pos, L, p["grid"], p["P"]
        self.xi, self.rc = p["xi"], p.get("rc", 0.0)
        self.h = L / self.n
        ms = 0.976 * math.sqrt(math.pi * self.P)
        self.alpha = 2.0 * ms * ms / (self.P * self.h) ** 2
        self._wave_setup()
        if real:
            self._real_setup()

    # ---- wave space
    def _wave_setup(self):
        n, L, dev = self.n, self.L, self.pos.device
        k1 = torch.arange(n, device=dev, dtype=torch.float64)
        k1 = torch.where(k1 <= n // 2, k1, k1 - n)
        kx = torch.arange(n // 2 + 1, device=dev, dtype=torch.float64)
        m2 = k1[:, None, None] ** 2 + k1[None, :, None] ** 2 + kx[None, None, :] ** 2
        k2 = m2 * (2 * math.pi / L) ** 2
        k2[0, 0, 0] = 1.0
        H = (1 + k2 / (4 * self.xi ** 2)) * torch.exp(-k2 / (4 * self.xi ** 2) + k2 / (2 * self.alpha)) / k2 / n ** 3
        H[0, 0, 0] = 0.0
        z = k2.sqrt()
        self.fm = z.sin() / z
        self.fd = torch.where(z < 1e-2, 1 - z * z / 10 + z ** 4 / 280, 3 * (z.sin() - z * z.cos()) / z ** 3)
        self.H, m2[0, 0, 0] = H, 1.0
        self.kv, self.m2 = (kx[None, None, :], k1[None, :, None], k1[:, None, None]), m2
        ar = torch.arange(self.P, device=dev)
        g = torch.floor(self.pos / self.h).long()[:, :, None] - self.P // 2 + 1 + ar
        self.y = g * self.h - self.pos[:, :, None]  # (N, 3, P)
        self.w = torch.exp(-self.alpha * self.y ** 2)
        self.g = g % n

    def _points(self, a, b):
        g, n = self.g[a:b], self.n
        at = (g[:, 2, :, None, None] * n + g[:, 1, None, :, None]) * n + g[:, 0, None, None, :]
        w, y = self.w[a:b], self.y[a:b]
        W = w[:, 2, :, None, None] * w[:, 1, None, :, None] * w[:, 0, None, None, :] * (self.alpha / math.pi) ** 1.5
        ys = (y[:, 0, None, None, :], y[:, 1, None, :, None], y[:, 2, :, None, None])
        return at, W, ys

    def wave(self, x):
        n, N, dev = self.n, len(self.pos), self.pos.device
        chunk = max(1, (1 << 24) // self.P ** 3)
        F = x[:, :3]
        D = _strain(x[:, 6:]) + 0.5 * _cross_matrix(x[:, 3:6])
        grid = torch.zeros(6, n ** 3, device=dev, dtype=torch.float64)
        for a in range(0, N, chunk):
            at, W, ys = self._points(a, a + chunk)
            at = at.reshape(-1)
            for c in range(3):
                grid[c].index_add_(0, at, (W * F[a:a + chunk, c, None, None, None]).reshape(-1))
                Dy = sum(D[a:a + chunk, c, e, None, None, None] * ys[e] for e in range(3))
                grid[3 + c].index_add_(0, at, (2 * self.alpha * W * Dy).reshape(-1))
        s = torch.fft.rfftn(grid.reshape(6, n, n, n), dim=(1, 2, 3))
        v = [self.H * (self.fm * s[c] + self.fd * s[3 + c]) for c in range(3)]
        kv = sum(self.kv[c] * v[c] for c in range(3)) / self.m2
        v = [v[c] - self.kv[c] * kv for c in range(3)]
        s = torch.stack([self.fm * u for u in v] + [self.fd * u for u in v])
        f = torch.fft.irfftn(s, s=(n, n, n), dim=(1, 2, 3), norm="forward").reshape(6, -1)
        out = torch.zeros(N, 11, device=dev, dtype=torch.float64)
        for a in range(0, N, chunk):
            at, W, ys = self._points(a, a + chunk)
            W = W * self.h ** 3
            G = torch.empty(len(W), 3, 3, device=dev, dtype=torch.float64)
            for c in range(3):
                out[a:a + chunk, c] = (W * f[c][at]).sum((1, 2, 3))
                Wd = 2 * self.alpha * W * f[3 + c][at]
                for e in range(3):
                    G[:, c, e] = (Wd * ys[e]).sum((1, 2, 3))
            out[a:a + chunk, 3:6] = 0.5 * torch.stack([G[:, 2, 1] - G[:, 1, 2], G[:, 0, 2] - G[:, 2, 0],
                                                       G[:, 1, 0] - G[:, 0, 1]], 1)
            out[a:a + chunk, 6:] = _five(G)
        return out

    # ---- real space
    def _radial(self, r):
        """Wave-part radial functions at r: (MM 1, MM 2, MD 2, MD 3, DD 2, DD 3, DD 4),
        (-1)^(n+1) / (2 pi^2) int H f_s f_t k^(2n-2) j_n(kr) / (kr)^n dk, with
        j_n(z)/z^n by its Poisson integral."""
        t, w = np.polynomial.legendre.leggauss(400)
        K = 2 * self.xi * math.sqrt(46.0)
        k, wk = 0.5 * K * (t + 1), 0.5 * K * w
        x = k * k / (4 * self.xi ** 2)
        H = (1 + x) * np.exp(-x) * wk
        fm = np.sin(k) / k
        fd = np.where(k < 1e-2, 1 - k * k / 10 + k ** 4 / 280, 3 * (np.sin(k) - k * np.cos(k)) / k ** 3)
        cos = np.cos(np.outer(r, k)[:, :, None] * t)
        out = []
        for ff, m in ((fm * fm, 1), (fm * fm, 2), (fm * fd, 2), (fm * fd, 3), (fd * fd, 2), (fd * fd, 3), (fd * fd, 4)):
            jn = cos @ (w * (1 - t * t) ** m) / (2 ** (m + 1) * math.factorial(m))
            out.append((1 if m % 2 else -1) * (jn @ (H * ff * k ** (2 * m - 2))) / (2 * math.pi ** 2))
        return np.stack(out)

    def _real_setup(self):
        pos, L, dev = self.pos, self.L, self.pos.device
        ii, jj = [], []
        for a in range(0, len(pos), 2048):
            d = pos[a:a + 2048, None, :] - pos[None, :, :]
            d -= L * torch.round(d / L)
            i, j = torch.nonzero(d.square().sum(2) < self.rc ** 2, as_tuple=True)
            ii.append(i + a)
            jj.append(j)
        i, j = torch.cat(ii), torch.cat(jj)
        keep = i != j
        self.i, self.j = i[keep], j[keep]
        # Chebyshev interpolation of the radial functions over [0, rc]
        m = 128
        th = np.pi * (np.arange(m) + 0.5) / m
        v = self._radial(0.5 * self.rc * (np.cos(th) + 1))
        c = torch.from_numpy(2.0 / m * (v @ np.cos(np.outer(th, np.arange(m))))).to(dev)
        c[:, 0] *= 0.5
        d = pos[self.i] - pos[self.j]
        self.d = d - L * torch.round(d / L)
        r = self.d.norm(dim=1)
        t = 2 * r / self.rc - 1
        b1 = b2 = torch.zeros(7, len(r), device=dev, dtype=torch.float64)
        for q in range(m - 1, 0, -1):
            b1, b2 = 2 * t * b1 - b2 + c[:, q, None], b1
        wave = t * b1 - b2 + c[:, 0, None]
        q, c8 = 1 / r, 1 / (8 * math.pi)
        free = torch.stack([q - 2 / 3 * q ** 3, -q ** 3 + 2 * q ** 5, -q ** 3 + 1.6 * q ** 5, 3 * q ** 5 - 8 * q ** 7,
                            -q ** 3 + 1.2 * q ** 5, 3 * q ** 5 - 6 * q ** 7, -15 * q ** 7 + 42 * q ** 9]) * c8
        self.ph = free - wave
        w0 = self._radial(np.zeros(1))[:, 0]
        self.self_ = (1 / (6 * math.pi) - 2 * w0[0], 1 / (8 * math.pi) + 2.5 * w0[4], 3 / (20 * math.pi) + 3 * w0[4])

    def real(self, x):
        out = torch.zeros(len(self.pos), 11, device=x.device, dtype=torch.float64)
        S = _strain(x[:, 6:])
        for a in range(0, len(self.i), 1 << 21):
            b = slice(a, a + (1 << 21))
            i, j, d = self.i[b], self.j[b], self.d[b]
            p1, p2, q2, q3, s2, s3, s4 = (v[:, None] for v in self.ph[:, b])
            F, T, Sj = x[j, :3], x[j, 3:6], S[j]
            Sx = (Sj @ d[:, :, None])[:, :, 0]
            r2 = d.square().sum(1, True)
            xF, xT, xSx = (d * F).sum(1, True), (d * T).sum(1, True), (d * Sx).sum(1, True)
            g, al, be = r2 * q3 + 5 * q2, r2 * s4 + 7 * s3, r2 * s3 + 5 * s2
            us = -(r2 * q3 + 3 * q2)
            dT = torch.linalg.cross(d, T)
            u = (r2 * p2 + 2 * p1) * F + (q3 * xSx - p2 * xF) * d + 0.5 * g * dT + us * Sx
            om = 0.5 * g * torch.linalg.cross(d, F) + 0.25 * al * xT * d + 0.25 * (be - al * r2 - 3 * be) * T \
                - 0.5 * al * torch.linalg.cross(d, Sx)
            v = -us * F + 0.5 * al * dT + (4 * s3 - al) * Sx + (s4 * xSx - q3 * xF) * d
            e = d[:, :, None] * v[:, None, :] + (2 * s2 - be)[:, :, None] * Sj
            out.index_add_(0, i, torch.cat([u, om, _five(e)], 1))
        t, r, s = self.self_
        return out + torch.cat([t * x[:, :3], r * x[:, 3:6], s * x[:, 6:]], 1)

    def __call__(self, x):
        return self.real(x) + self.wave(x)


class _Saddle:
    """[M, B Sigma^T; Sigma B^T, -R] with the pair lubrication (gap clamp 1e-3)."""

    def __init__(self, pos, body, L, p):
        self.M, self.N, self.body = _Mobility(pos, L, p), len(pos), body.long()
        self.nbody = int(body.max()) + 1
        cnt = torch.zeros(self.nbody, 1, device=pos.device, dtype=torch.float64).index_add_(
            0, self.body, torch.ones(self.N, 1, device=pos.device, dtype=torch.float64))
        self.X = torch.zeros(self.nbody, 3, device=pos.device, dtype=torch.float64).index_add_(0, self.body, pos) / cnt
        self.lever = pos - self.X[self.body]
        # lubrication pairs among the mobility's (cut-off 3 < R_c)
        i, j, d, rl = self.M.i, self.M.j, -self.M.d, p["lub_cutoff"]
        r = d.norm(dim=1)
        k = (r < rl) & (self.body[i] != self.body[j])
        self.i, self.j, self.r = i[k], j[k], r[k][:, None]
        self.nn = d[k] / self.r
        if len(self.i):
            e, ec = (self.r - 2).clamp(min=1e-3), rl - 2
            q = 0.25 / e - 0.225 * e.log()
            self.A = 6 * math.pi * (q - (0.25 / ec - 0.225 * math.log(ec))).clamp(min=0)
            self.B = math.pi * (math.log(ec) - e.log()).clamp(min=0)
            self.D = 0.8 * self.B
        self._block(p["precond_cutoff"])

    def near(self, U, E):
        """Near-field bead forces, torques (N, 6) and stresslets (N, 3, 3)."""
        F = torch.zeros(self.N, 6, device=U.device, dtype=torch.float64)
        S = torch.zeros(self.N, 3, 3, device=U.device, dtype=torch.float64)
        if len(self.i):
            om = U[self.body, 3:]
            du = U[self.body, :3] + torch.linalg.cross(om, self.lever) - self.lever @ E
            i, j, n, r = self.i, self.j, self.nn, self.r
            s = du[j] - du[i] + 0.5 * r * torch.linalg.cross(n, om[i] + om[j]) + r * (n @ E)
            ns = (n * s).sum(1, True)
            Gs = self.A * ns * n + self.B * (s - ns * n)
            t = om[i] - om[j]
            tq = 0.5 * r * torch.linalg.cross(n, Gs) - self.D * (t - (n * t).sum(1, True) * n)
            F.index_add_(0, i, torch.cat([Gs, tq], 1))
            sn = 0.25 * r[:, :, None] * (Gs[:, :, None] * n[:, None, :] + n[:, :, None] * Gs[:, None, :])
            S.index_add_(0, i, sn)
        return F, S

    def gather(self, f):
        f = torch.cat([f[:, :3], f[:, 3:6] + torch.linalg.cross(self.lever, f[:, :3].contiguous())], 1)
        return torch.zeros(self.nbody, 6, device=f.device, dtype=torch.float64).index_add_(0, self.body, f)

    def rigid(self, U):
        om = U[self.body, 3:]
        u = U[self.body, :3] + torch.linalg.cross(om, self.lever)
        return torch.cat([u, om, torch.zeros(self.N, 5, device=U.device, dtype=torch.float64)], 1)

    def split(self, x):
        return x[:11 * self.N].reshape(-1, 11), x[11 * self.N:].reshape(-1, 6)

    def __call__(self, x):
        f, U = self.split(x)
        none = torch.zeros(3, 3, device=x.device, dtype=torch.float64)
        y2 = self.gather(f[:, :6]) + self.gather(self.near(U, none)[0])
        return torch.cat([(self.M(f) + self.rigid(U)).reshape(-1), y2.reshape(-1)])

    def _block(self, rp):
        z = 6 * math.pi
        eye = torch.eye(3, device=self.lever.device, dtype=torch.float64)
        R = z * torch.eye(6, device=self.lever.device, dtype=torch.float64).repeat(self.N, 1, 1)
        if len(self.i):
            k = (self.r < rp)[:, 0]
            n, r, A, B, D = self.nn[k], self.r[k][:, :, None], self.A[k][:, :, None], self.B[k][:, :, None], self.D[k][:, :, None]
            nn = n[:, :, None] * n[:, None, :]
            Nx = _cross_matrix(n)
            top = torch.cat([A * nn + B * (eye - nn), -0.5 * r * B * Nx], 2)
            low = torch.cat([0.5 * r * B * Nx, (0.25 * r * r * B + D) * (eye - nn)], 2)
            R.index_add_(0, self.i[k], torch.cat([top, low], 1))
        Sg = torch.eye(6, device=R.device, dtype=torch.float64).repeat(self.N, 1, 1)
        Sg[:, 3:, :3] = _cross_matrix(self.lever)
        Bm = torch.zeros(self.nbody, 6, 6, device=R.device, dtype=torch.float64)
        self.Binv = torch.linalg.inv(Bm.index_add_(0, self.body, Sg @ R @ Sg.transpose(1, 2)))

    def precond(self, r):
        z = 6 * math.pi
        r1, r2 = self.split(r)
        u = -(self.Binv @ (r2 - z * self.gather(r1[:, :6]))[:, :, None])[:, :, 0]
        return torch.cat([(z * (r1 - self.rigid(u))).reshape(-1), u.reshape(-1)])

    def solve(self, b, tol=1e-10, most=200):
        beta = b.norm()
        V, Z, H = [b / beta], [], np.zeros((most + 1, most))
        e1 = np.zeros(most + 1)
        e1[0] = float(beta)
        for k in range(most):
            Z.append(self.precond(V[k]))
            w = self(Z[k])
            Q = torch.stack(V)
            for _ in range(2):
                h = Q @ w
                w = w - h @ Q
                H[:k + 1, k] += h.cpu().numpy()
            H[k + 1, k] = float(w.norm())
            V.append(w / H[k + 1, k])
            y = np.linalg.lstsq(H[:k + 2, :k + 1], e1[:k + 2], rcond=None)[0]
            if np.linalg.norm(H[:k + 2, :k + 1] @ y - e1[:k + 2]) < tol * float(beta):
                break
        return torch.from_numpy(y).to(b) @ torch.stack(Z)

    def motion(self, ft, shear):
        """Velocities (U, Omega) and stresslets of the aggregates."""
        E = torch.zeros(3, 3, device=ft.device, dtype=torch.float64)
        E[0, 1] = E[1, 0] = 0.5 * shear
        zero = torch.zeros(self.nbody, 6, device=ft.device, dtype=torch.float64)
        b1 = torch.zeros(self.N, 11, device=ft.device, dtype=torch.float64)
        b1[:, :3] = self.lever @ E
        b1[:, 6:] = _five(E[None])
        x = self.solve(torch.cat([b1.reshape(-1), -(ft + self.gather(self.near(zero, E)[0])).reshape(-1)]))
        f, U = self.split(x)
        fn, sn = self.near(U, E)
        force = f[:, :3] + fn[:, :3]
        rf = 0.5 * (self.lever[:, :, None] * force[:, None, :] + force[:, :, None] * self.lever[:, None, :])
        S = torch.zeros(self.nbody, 3, 3, device=ft.device, dtype=torch.float64).index_add_(
            0, self.body, _strain(f[:, 6:] + _five(sn)) + rf)
        vel = U.clone()
        vel[:, 0] += shear * self.X[:, 1]
        vel[:, 5] -= 0.5 * shear
        return vel, S


def exact(case, seed):
    """Operator applications and solves of up to about 15 000 beads; the larger
    ones, the random terms and the batch would take too long here or have no
    independent value."""
    call = case["call"]
    if call in ("batch", "brownian", "step"):
        return None
    st = prepare(case, seed)
    if call == "wave":
        p = {"grid": case["grid"], "P": case["P"], "xi": case["xi"]}
        return [_Mobility(st["pos"], st["L"], p, real=False).wave(st["x"])]
    s, pos, body, L = st["s"], st["pos"], st["body"], st["L"]
    p = s.params
    if call == "forces":
        return [_pair_forces(pos, body, L)]
    if s.n_beads > 15000:
        return None
    if call == "mobility":
        return [_Mobility(pos, L, p)(st["x"].reshape(-1, 11)).reshape(-1)]
    A = _Saddle(pos, body, L, p)
    if call == "saddle":
        return [A(st["x"])]
    # the call stops at its own tolerance, this one far below it
    return list(A.motion(st["ft"], 1.0)) if s.n_beads <= 4500 else None


def _pair_forces(pos, body, L, kn=2.5e3, hamaker=15.0, zeta=4.0, kappa=1.0, h_c=0.03, r_cut=5.0):
    """Hertz and DLVO pair forces summed to aggregate forces and torques."""
    N, nb, b = len(pos), int(body.max()) + 1, body.long()
    X = torch.zeros(nb, 3, device=pos.device, dtype=torch.float64).index_add_(0, b, pos)
    X = X / torch.bincount(b, minlength=nb).double()[:, None]
    out = torch.zeros(nb, 6, device=pos.device, dtype=torch.float64)
    for a in range(0, N, 1024):
        d = pos[a:a + 1024, None, :] - pos[None, :, :]
        d -= L * torch.round(d / L)
        r = d.norm(dim=2)
        i, j = torch.nonzero((r < r_cut) & (b[a:a + 1024, None] != b[None, :]), as_tuple=True)
        d, r, i = d[i, j], r[i, j], i + a
        rv = r.clamp(min=2.0) + h_c
        q = rv * rv - 4.0
        f = kn * (2.0 - r).clamp(min=0.0) ** 1.5
        f = f + hamaker / 6 * (-4 * rv / q ** 2 - 4 / rv ** 3 + 2 * rv / q - 2 / rv)
        f = f + zeta * torch.exp(-kappa * (r - 2.0)) * (1 / r ** 2 + kappa / r)
        F = (f / r)[:, None] * d
        out.index_add_(0, b[i], torch.cat([F, torch.linalg.cross(pos[i] - X[b[i]], F)], 1))
    return out
