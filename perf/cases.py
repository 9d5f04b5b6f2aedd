"""Measured cases of the MHD framework: what is timed, on which inputs, and
the plain FP64 result each case is held against.

A case is one pass a user's program makes through the public Python API with a
new state on the device (or, for the batch, in host memory): hand the state to
the box, advance it by a number of double steps with the time step chosen by
the CFL condition on the device, and take the new state back.  The sizes come
from the paper's test problems, the benchmark and the batch generator of this
repository, with odd and flat boxes added; `draw` spreads over the same ranges.

`exact` is the method written once more with plain FP64 torch arithmetic on
whole arrays (no code of the package is used by it).
"""
import math

import numpy as np
import torch

import paper_0910_2854_gb300 as F
from paper_0910_2854_gb300 import workloads as W
from paper_0910_2854_gb300.decomp import SlabRun, slab_extent

CFL = 0.4
DEVICE = "cuda"
PERIODIC, OUTFLOW = 0, 1
VANLEER, MINMOD, HYBRID = 0, 1, 3


def _box(name, dims, steps, precision="fp32", init="smooth", bc=PERIODIC, limiter=VANLEER, physics="plain",
         monitor=False, kind="box"):
    nx, ny, nz = dims
    return {"name": name, "kind": kind, "nx": nx, "ny": ny, "nz": nz, "steps": steps, "precision": precision,
            "init": init, "bc": bc, "limiter": limiter, "physics": physics, "monitor": monitor}


def listed():
    return [
        # The paper's circularly polarised Alfven wave on its small box in
        # double precision: the check run, bound by launches and latency.
        _box("alfven_32_fp64", (32, 32, 32), 10, "fp64", "alfven"),
        # A small single-precision box, one of many in a parameter scan.
        _box("smooth_48x40x36_fp32", (48, 40, 36), 10),
        # The paper's two-dimensional rotor: a flat box of one cell along z.
        _box("rotor_256x256x1_fp32", (256, 256, 1), 10, init="rotor", bc=OUTFLOW),
        # Ragged odd extents with open boundaries and the minmod limiter.
        _box("ragged_101x67x83_fp32", (101, 67, 83), 4, bc=OUTFLOW, limiter=MINMOD),
        # Turbulence at an ordinary size, with the diagnostics read after the
        # steps as a run's log does.
        _box("turbulence_256_fp32", (256, 256, 256), 4, init="turbulence", monitor=True),
        # Turbulence at a production size (the state is far larger than L2).
        _box("turbulence_640_fp32", (640, 640, 640), 2, init="turbulence"),
        # The Orszag-Tang-type vortex of the benchmark in double precision.
        _box("orszag_tang_256_fp64", (256, 256, 256), 1, "fp64", "orszag_tang"),
        # A star in hydrostatic equilibrium: unsplit gravity with the
        # hydrostatic-gradient correction, open boundaries.
        _box("polytrope_192_hse_fp32", (192, 192, 192), 2, init="polytrope", bc=OUTFLOW, physics="hse"),
        # An irregular Cartesian mesh.
        _box("stretched_160x128x96_fp32", (160, 128, 96), 2, physics="mesh"),
        # Operator-split gravity in double precision, uneven box.
        _box("split_gravity_72x60x51_fp64", (72, 60, 51), 2, "fp64", limiter=MINMOD, physics="split"),
        # One rank's part of a box split into z-slabs: ghost planes exchanged
        # before every operator, operators launched one by one.
        _box("slab_160x128x64_fp32", (160, 128, 64), 1, kind="slab"),
        # A parameter study: uneven shock-tube and blast boxes advanced
        # together; this API takes and returns host arrays.
        {"name": "batch_12_fp32", "kind": "batch", "boxes": 12, "smallest": 32, "largest": 96, "steps": 20,
         "precision": "fp32"},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("fp32", "fp32", "fp32", "fp64", "fp64", "slab", "batch"))
    if kind == "batch":
        lo = 2 * size(8, 24)
        return {"kind": "batch", "boxes": rng.randint(3, 12), "smallest": lo, "largest": lo + 2 * size(4, 24),
                "steps": rng.randint(2, 20), "precision": "fp32"}
    if kind == "slab":
        c = _box("", (size(24, 192), size(24, 192), size(16, 96)), 1, kind="slab",
                 limiter=rng.choice((VANLEER, MINMOD)))
    else:
        most = 24e6 if kind == "fp32" else 4e6
        while True:
            dims = (size(12, 400), size(12, 400), size(1, 400))
            if rng.random() < 0.5:  # even fast extents are the common case
                dims = tuple(d + d % 2 for d in dims)
            if dims[0] * dims[1] * dims[2] <= most:
                break
        cells = dims[0] * dims[1] * dims[2]
        c = _box("", dims, max(1, min(rng.randint(1, 10), int(most / cells))), kind,
                 bc=rng.choice((PERIODIC, OUTFLOW)),
                 limiter=rng.choice((VANLEER, VANLEER, MINMOD, HYBRID)),
                 physics=rng.choice(("plain", "plain", "plain", "unsplit", "split", "hse", "mesh")))
        if c["physics"] == "hse" and c["limiter"] == HYBRID:
            c["limiter"] = VANLEER
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _modes(rng, dims, pos, amp, count=4):
    """Sum of a few Fourier modes at tensor-product points, pos[a] the offset
    of the points from the lower cell faces in cells along axis a."""
    t = [torch.arange(n, dtype=torch.float64, device=DEVICE).add_(pos[a]).mul_(2.0 * math.pi / n)
         for a, n in enumerate(dims)]
    out = torch.zeros((dims[2], dims[1], dims[0]), dtype=torch.float64, device=DEVICE)
    for _ in range(count):
        k = [int(v) for v in rng.randint(-2, 3, size=3)]
        a, ph = rng.uniform(0.3, 1.0) * amp, rng.uniform(0.0, 2.0 * math.pi)
        zy = (k[2] * t[2])[:, None] + (k[1] * t[1])[None, :] + ph
        x = k[0] * t[0]
        out.addcmul_(a * torch.sin(zy)[:, :, None], torch.cos(x))
        out.addcmul_(a * torch.cos(zy)[:, :, None], torch.sin(x))
    return out


def _lower(a, axis, bc):
    """a at the next lower index along axis (0 = x): the periodic image, or a
    copy of the first entry."""
    dim = 2 - axis
    if bc == PERIODIC:
        return torch.roll(a, 1, dim)
    return torch.cat([a.narrow(dim, 0, 1), a.narrow(dim, 0, a.shape[dim] - 1)], dim)


def _assemble(rho, v, p, b, gamma, bc):
    q = torch.empty((8,) + tuple(rho.shape), dtype=torch.float64, device=rho.device)
    q[0] = rho
    q[4] = p / (gamma - 1.0)
    for a in range(3):
        q[1 + a] = rho * v[a]
        q[4] += 0.5 * rho * v[a] * v[a]
        q[5 + a] = b[a]
    for a in range(3):
        q[4] += 0.5 * (0.5 * (_lower(q[5 + a], a, bc) + q[5 + a])) ** 2
    return q


def _smooth(dims, h, bc, seed, gamma=5.0 / 3.0):
    """Smooth flow, Mach number about 0.5, divergence-free field."""
    rng = np.random.RandomState(seed % (1 << 31))
    rho = 1.0 + _modes(rng, dims, (0.5, 0.5, 0.5), 0.1)
    p = 1.0 + _modes(rng, dims, (0.5, 0.5, 0.5), 0.1)
    v = [_modes(rng, dims, (0.5, 0.5, 0.5), 0.25) for _ in range(3)]
    L = [dims[a] * h[a] / (2.0 * math.pi) for a in range(3)]
    A = []
    for a in range(3):
        pos = [1.0, 1.0, 1.0]
        pos[a] = 0.5
        A.append(_modes(rng, dims, pos, 0.1 * min(L)))
    b = []
    for a in range(3):
        c, d = (a + 1) % 3, (a + 2) % 3
        b.append((0.2, 0.1, 0.05)[a] + (A[d] - _lower(A[d], c, PERIODIC)) / h[c]
                 - (A[c] - _lower(A[c], d, PERIODIC)) / h[d])
    return _assemble(rho, v, p, b, gamma, bc)


def _widths(dims, h, seed):
    out = []
    for a, n in enumerate(dims):
        x = (np.arange(n) + 0.5) / n
        w = 1.0 + (0.25 + 0.05 * a) * np.sin(2.0 * math.pi * x + 0.3 * (seed % 17) + 0.7 * a)
        out.append(n * h[a] * w / w.sum())
    return out


def _problem(case, seed):
    """State (FP64, on the device) and parameters of a box case."""
    dims = (case["nx"], case["ny"], case["nz"])
    rng = np.random.RandomState((seed * 7919 + 13) % (1 << 31))
    gamma, phi, widths = 5.0 / 3.0, None, None
    h = tuple(1.0 / n for n in dims)
    if case["init"] == "alfven":
        w = W.alfven_x(dims[0], dims[1], dims[2], amp=float(rng.uniform(0.05, 0.15)))
        q, gamma, h = torch.as_tensor(w.state, device=DEVICE), w.gamma, w.h
    elif case["init"] == "rotor":
        w = W.rotor(dims[0], r0=float(rng.uniform(0.09, 0.11)), r1=float(rng.uniform(0.115, 0.13)))
        q, gamma, h = torch.as_tensor(w.state, device=DEVICE), w.gamma, w.h
    elif case["init"] == "turbulence":
        w = W.turbulence(dims[0], seed_v=910285 + seed % 100000, seed_a=1910286 + seed % 100000, device=DEVICE,
                         dtype=torch.float32)
        q, gamma, h = w.state, w.gamma, w.h
    elif case["init"] == "orszag_tang":
        # the vortex at a random offset along each axis
        x, y, z = [2.0 * math.pi * ((torch.arange(n, dtype=torch.float64, device=DEVICE) + 0.5) / n
                                    + rng.uniform()) for n in dims]
        one = torch.ones((dims[2], dims[1], dims[0]), dtype=torch.float64, device=DEVICE)
        X, Y, Z = one * x, one * y[:, None], one * z[:, None, None]
        s = 1.0 / math.sqrt(4.0 * math.pi)
        q = _assemble(one * (25.0 / (36.0 * math.pi)), (-torch.sin(Y), torch.sin(X), 0.1 * torch.sin(Z)),
                      one * (5.0 / (12.0 * math.pi)), (-s * torch.sin(Y), s * torch.sin(2.0 * X), 0.0 * one), gamma,
                      case["bc"])
    elif case["init"] == "polytrope":
        # n = 1 star with a weak random flow and field, see workloads.polytrope
        gamma, wd = 2.0, 1.45
        h = tuple(2.0 * wd / n for n in dims)
        K, M, atm = 2.0 / math.pi, 4.0 / math.pi, 1e-3
        xs = [-wd + (torch.arange(n, dtype=torch.float64, device=DEVICE) + 0.5) * h[a] for a, n in enumerate(dims)]
        r = torch.sqrt(xs[2][:, None, None] ** 2 + xs[1][:, None] ** 2 + xs[0] ** 2)
        prof = torch.sinc(r)
        rho = torch.where(r < 1.0, prof.clamp(min=atm), torch.full_like(r, atm))
        p = (K * rho * rho).clamp(min=atm * K)
        phi = torch.where(r < 1.0, -2.0 * K * prof - M, -M / r).cpu().numpy()
        v = [_modes(rng, dims, (0.5, 0.5, 0.5), 0.01) for _ in range(3)]
        zero = torch.zeros_like(r)
        q = _assemble(rho, v, p, (zero, zero, zero), gamma, case["bc"])
    else:
        q = _smooth(dims, h, case["bc"], seed)
        if case["physics"] in ("unsplit", "split", "hse"):
            phi = _modes(rng, dims, (0.5, 0.5, 0.5), 0.1).cpu().numpy()
        if case["physics"] == "mesh":
            widths = _widths(dims, h, seed)
    dtype = torch.float32 if case["precision"] == "fp32" else torch.float64
    return q.to(dtype), gamma, h, phi, widths


def _moving_blast(dims, rng):
    """A blast in a moving gas, its edge a few cells wide (a sharp sphere at
    rest leaves velocities of rounding size in its middle, whose sign picks
    the upwind cell of the field)."""
    w = W.blast(*dims)
    r2 = np.zeros((dims[2], dims[1], dims[0]))
    for a, c in enumerate(rng.uniform(0.42, 0.47, size=3)):
        x = ((np.arange(dims[a]) + 0.5) / dims[a] - c) * dims[a] * w.h[a]
        r2 = r2 + (x * x).reshape([-1 if k == 2 - a else 1 for k in range(3)])
    size = min(dims) * w.h[0]
    p = 1.0 + rng.uniform(10.0, 30.0) * 0.5 * (1.0 - np.tanh((np.sqrt(r2) / size - 0.2) / 0.06))
    v = rng.uniform(0.3, 0.8, size=3)
    w.state[4] = p / (w.gamma - 1.0) + 0.5 * np.sum(v * v) + 0.5
    for a in range(3):
        w.state[1 + a] = v[a]
    return w


def _batch_boxes(case, seed):
    """Uneven shock tubes and off-centre blasts, host states in FP64."""
    rng = np.random.RandomState((seed * 104729 + 7) % (1 << 31))
    lo, hi = case["smallest"], case["largest"]
    shapes = np.random.RandomState(2009 + case["boxes"])  # the shapes belong to the case, the values to the seed
    out = []
    for k in range(case["boxes"]):
        dims = tuple(2 * int(v) for v in shapes.randint(lo // 2, hi // 2 + 1, size=3))
        kind, axis = ("sod", "brio_wu", "blast")[k % 3], int(shapes.randint(0, 3))
        if kind == "blast":
            w = _moving_blast(dims, rng)
        else:
            w = W.batch_box(kind, dims, axis)
            w.state[0] *= rng.uniform(0.9, 1.1)
            # a field across the tube (constant, so divergence-free) and its energy
            c = 5 + (axis + 2) % 3
            add = float(rng.uniform(0.02, 0.1))
            w.state[4] += 0.5 * ((w.state[c] + add) ** 2 - w.state[c] ** 2)
            w.state[c] += add
        out.append(w)
    return out


def prepare(case, seed):
    if case["kind"] == "batch":
        ws = _batch_boxes(case, seed)
        batch = F.Batch([w.dims for w in ws], [w.gamma for w in ws], [w.bc for w in ws], [w.h for w in ws])
        return {"kind": "batch", "batch": batch, "states": [w.state for w in ws], "steps": case["steps"]}
    q, gamma, h, phi, widths = _problem(case, seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    lo = hi = 0
    if case["kind"] == "slab":
        _, _, lo, hi = slab_extent(nz, 0, 1, True)
        q = torch.cat([q[:, nz - lo:], q, q[:, :hi]], 1).contiguous()
        h = (h[0], h[1], h[2])
    phys = case["physics"]
    box = F.Box(nx, ny, nz + lo + hi, gamma, bc=case["bc"], precision=case["precision"], limiter=case["limiter"],
                hse=phys == "hse", gravity="split" if phys == "split" else "unsplit", h=h)
    if phi is not None:
        box.set_potential(phi)
    if widths is not None:
        box.set_mesh(widths)
    s = {"kind": case["kind"], "box": box, "q": q, "out": torch.empty_like(q), "steps": case["steps"],
         "monitor": case["monitor"], "lo": lo, "nk": nz}
    if case["kind"] == "slab":
        s["slab"] = SlabRun(box, nx, ny, nz, 0, 1, True, device=DEVICE, dtype=q.dtype)
    return s


def run(s):
    if s["kind"] == "batch":
        b = s["batch"]
        for k, q in enumerate(s["states"]):
            b.set_state(k, q)
        b.step(CFL, s["steps"])
        return {"states": [b.get_state(k) for k in range(len(s["states"]))], "dt": b.last_dt()}
    box = s["box"]
    box.set_state(s["q"])
    if s["kind"] == "slab":
        dt = s["slab"].step_cfl(CFL, s["steps"])
        return {"state": box.get_state_device(s["out"])[:, s["lo"]:s["lo"] + s["nk"]], "dt": dt}
    box.step_cfl(CFL, s["steps"])
    r = {"state": box.get_state_device(s["out"]), "dt": box.last_dt()}
    if s["monitor"]:
        r["totals"] = box.diagnostics()[:8]
    return r


# ---------------------------------------------------------------------------
# work and tolerance
# ---------------------------------------------------------------------------
# Arithmetic of one double step per cell: six sweeps of the fluid operator
# (two cell evaluations of about 70 operations, 25 for the first-order flux,
# 130 for the limited one, 25 for the two updates) and six of the magnetic one
# (two transverse face pencils of about 45 operations, 6 for the constraint).
FLOPS_PER_CELL_STEP = 6 * (2 * 70 + 25 + 130 + 25 + 2 * 45 + 6)


def _cells(case):
    if case["kind"] == "batch":
        shapes = np.random.RandomState(2009 + case["boxes"])
        total = 0
        for _ in range(case["boxes"]):
            d = [2 * int(v) for v in shapes.randint(case["smallest"] // 2, case["largest"] // 2 + 1, size=3)]
            shapes.randint(0, 3)
            total += d[0] * d[1] * d[2]
        return total
    return case["nx"] * case["ny"] * case["nz"]


def work(case):
    """Bytes: the state read once and written once.  A pass of n steps needs
    no more than that where the state fits the caches; a state larger than
    they are also moves once through memory per step."""
    cells = _cells(case)
    size = 4 if case["precision"] == "fp32" else 8
    once = 16.0 * size * cells
    passes = case["steps"] if 8.0 * size * cells > 128e6 else 1
    return {"bytes": once * passes, "flops": float(FLOPS_PER_CELL_STEP) * cells * case["steps"]}


def tolerance(case):
    """About four times the largest distance from `exact` seen over the listed
    cases and some sixty drawn ones (rel 2.6e-16 and 2.9e-7).  The largest
    single difference is set by cells where rounding picks another limiter
    branch or upwind cell (6e-15 and 6e-4 seen)."""
    if case["precision"] == "fp64":
        return {"rel": 1.1e-15, "max": 1e-12}
    return {"rel": 1.2e-6, "max": 2e-3}


# ---------------------------------------------------------------------------
# the method in plain FP64 torch
# ---------------------------------------------------------------------------
G = 4  # ghost cells of a sweep


def _ghosts(n, bc, device, lo=G, hi=G):
    s = torch.arange(-lo, n + hi, device=device)
    return s % n if bc == PERIODIC else s.clamp(0, n - 1)


def _limit(lim, a, b):
    if lim == MINMOD:
        return 0.5 * (torch.sign(a) + torch.sign(b)) * torch.minimum(a.abs(), b.abs())
    ab = a * b
    return torch.where(ab > 0, 2.0 * ab / torch.where(ab > 0, a + b, torch.ones_like(a)), torch.zeros_like(a))


def _centred(q, bc):
    return [0.5 * (_lower(q[5 + a], a, bc) + q[5 + a]) for a in range(3)]


def _speeds(rho, m, E, b, d, gamma):
    """velocity, pressure, b^2/2, sound and fast speed along d."""
    v = [m[a] / rho for a in range(3)]
    mag = 0.5 * (b[0] * b[0] + b[1] * b[1] + b[2] * b[2])
    p = (gamma - 1.0) * (E - 0.5 * (m[0] * v[0] + m[1] * v[1] + m[2] * v[2]) - mag)
    a2 = gamma * p / rho
    bt2 = (2.0 * mag - b[d] * b[d]) / rho
    B2 = b[d] * b[d] / rho + bt2
    cf = torch.sqrt(0.5 * (a2 + B2 + torch.sqrt((a2 - B2) ** 2 + 4.0 * a2 * bt2)))
    return v, p, mag, torch.sqrt(a2), cf


class _Cells:
    """Fluxes and speeds of a row of cells along d; u = (rho, m_x, m_y, m_z, E)."""

    def __init__(self, u, b, d, gamma):
        v, p, mag, self.cs, self.cf = _speeds(u[0], u[1:4], u[4], b, d, gamma)
        self.u, self.p, self.vn = u, p, v[d]
        self.F = [u[1 + d]]
        for a in range(3):
            f = u[1 + a] * v[d] - b[d] * b[a]
            self.F.append(f + p + mag if a == d else f)
        bv = b[0] * v[0] + b[1] * v[1] + b[2] * v[2]
        self.F.append((u[4] + p + mag) * v[d] - b[d] * bv)


def _hse_jump(c, phi, R, k):
    """Hydrostatic-corrected jump of component k across each interface."""
    x = c.u[k] + c.p if k == 4 else c.u[k]
    fac = (R(phi) - _L(phi, R)) / (_L(c.cs, R) * R(c.cs))
    du = R(c.u[k]) - _L(c.u[k], R)
    return du, _limit(MINMOD, du + 0.5 * (R(x) + _L(x, R)) * fac, du)


def _L(a, R):
    return a.narrow(R.dim, 0, a.shape[R.dim] - 1)


class _Right:
    """The right neighbours along a dimension (all entries but the first)."""

    def __init__(self, dim):
        self.dim = dim

    def __call__(self, a):
        return a.narrow(self.dim, 1, a.shape[self.dim] - 1)


def _fluid(q, d, dt, P):
    gamma, bc, h, lim, phys = P["gamma"], P["bc"], P["h"], P["limiter"], P["physics"]
    n, dim = q.shape[3 - d], 2 - d
    ix = _ghosts(n, bc, q.device)
    pick = lambda a: a.index_select(dim, ix)  # noqa: E731
    R = _Right(dim)
    inner = lambda a, k: a.narrow(dim, k, a.shape[dim] - 2 * k)  # noqa: E731
    u = [pick(q[k]) for k in range(5)]
    b = [pick(c) for c in _centred(q, bc)]
    shape = [1, 1, 1]
    shape[dim] = -1
    wd = None
    if P["widths"] is not None:
        wd = P["widths"][d].index_select(0, ix).view(shape)
    phi = pick(P["phi"]) if P["phi"] is not None and phys in ("unsplit", "hse") else None
    if phi is None and phys == "hse":
        phi = torch.zeros_like(u[0])
    c = _Cells(u, b, d, gamma)
    # predictor
    f1 = []
    for k in range(5):
        mean = 0.5 * (_L(c.F[k], R) + R(c.F[k]))
        if phys == "hse":
            du, dd = _hse_jump(c, phi, R, k)
            Da = torch.maximum(_L(c.vn, R).abs(), R(c.vn).abs())
            f1.append(mean - 0.5 * Da * du - 0.5 * torch.maximum(_L(c.cf, R), R(c.cf)) * dd)
        else:
            s = c.vn.abs() + c.cf
            f1.append(mean - 0.5 * torch.maximum(_L(s, R), R(s)) * (R(c.u[k]) - _L(c.u[k], R)))
    lam = dt / inner(wd, 1) if wd is not None else dt / h[d]
    up = [inner(u[k], 1) - 0.5 * lam * (R(f1[k]) - _L(f1[k], R)) for k in range(5)]
    del f1
    if phi is not None:
        span = 0.5 * wd.narrow(dim, 0, n + 2 * G - 2) + inner(wd, 1) + 0.5 * wd.narrow(dim, 2, n + 2 * G - 2) \
            if wd is not None else 2.0 * h[d]
        dphi = (phi.narrow(dim, 2, n + 2 * G - 2) - phi.narrow(dim, 0, n + 2 * G - 2)) / span
        up[1 + d] = up[1 + d] - 0.5 * dt * inner(u[0], 1) * dphi
        up[4] = up[4] - 0.5 * dt * inner(u[1 + d], 1) * dphi
    b1 = [inner(a, 1) for a in b]
    del c
    c = _Cells(up, b1, d, gamma)
    # corrector: interfaces between predicted cells e and e+1, e from the second
    m = n + 2 * G - 2
    mid = lambda a: a.narrow(dim, 1, m - 3)  # noqa: E731  (interface values of the middle ones)
    le, ri = (lambda a: a.narrow(dim, 1, m - 3)), (lambda a: a.narrow(dim, 2, m - 3))
    w1 = inner(wd, 1) if wd is not None else None
    limit = lim
    if lim == HYBRID:
        fast = (le(c.vn).abs() > le(c.cs)) | (ri(c.vn).abs() > ri(c.cs))
    un = []
    if phys == "hse":
        Da, Dc = torch.maximum(le(c.vn).abs(), ri(c.vn).abs()), torch.maximum(le(c.cf), ri(c.cf))
        phi1 = inner(phi, 1)
    else:
        s = c.vn.abs() + c.cf
        D = torch.maximum(le(s), ri(s))
    for k in range(5):
        dF = R(c.F[k]) - _L(c.F[k], R)
        three = lambda a: (a.narrow(dim, 0, m - 3), mid(a), a.narrow(dim, 2, m - 3))  # noqa: E731
        if phys == "hse":
            du, dd = _hse_jump(c, phi1, R, k)
            qs = [Da * x + Dc * y for x, y in zip(three(du), three(dd))]
        else:
            qs = [D * x for x in three(R(c.u[k]) - _L(c.u[k], R))]
        dFs = three(dF)
        args = [0.5 * (dFs[0] + qs[0]), 0.5 * (dFs[1] + qs[1]), 0.5 * (dFs[1] - qs[1]), 0.5 * (dFs[2] - qs[2])]
        sp = sm = 1.0
        if wd is not None:
            gap = 0.5 * (_L(w1, R) + R(w1))
            g = three(gap)
            args = [args[0] / g[0], args[1] / g[1], args[2] / g[1], args[3] / g[2]]
            sp, sm = le(w1), ri(w1)
        if lim == HYBRID:
            slp = torch.where(fast, _limit(MINMOD, args[0], args[1]), _limit(VANLEER, args[0], args[1]))
            slm = torch.where(fast, _limit(MINMOD, args[2], args[3]), _limit(VANLEER, args[2], args[3]))
        else:
            slp, slm = _limit(limit, args[0], args[1]), _limit(limit, args[2], args[3])
        f2 = 0.5 * (le(c.F[k]) + ri(c.F[k])) - 0.5 * qs[1] + 0.5 * (sp * slp - sm * slm)
        f2 = f2.narrow(dim, G - 3, n + 1)
        lo_ = dt / P["widths"][d].view(shape) if wd is not None else dt / h[d]
        un.append(q[k] - lo_ * (R(f2) - _L(f2, R)))
    if phi is not None:
        core = lambda a: a.narrow(dim, G - 1, n)  # noqa: E731
        un[1 + d] = un[1 + d] - dt * core(up[0]) * core(dphi)
        un[4] = un[4] - dt * core(up[1 + d]) * core(dphi)
    return torch.cat([torch.stack(un), q[5:]])


def _kick(q, d, tau, P):
    """Operator-split gravity: momentum along d and its kinetic energy."""
    n, dim = q.shape[3 - d], 2 - d
    i = _ghosts(n, P["bc"], q.device, 1, 1)
    ph = P["phi"].index_select(dim, i)
    m = q[1 + d] - tau * q[0] * (ph.narrow(dim, 2, n) - ph.narrow(dim, 0, n)) / (2.0 * P["h"][d])
    q = q.clone()
    q[4] += 0.5 * (m * m - q[1 + d] ** 2) / q[0]
    q[1 + d] = m
    return q


def _edge_fluxes(q, d, c, dt, P):
    """Fluxes of b_c along d at the edges, on the faces -1 .. n_c - 1 along c
    and the interfaces -1 .. n_d - 1 along d."""
    bc, lim = P["bc"], P["limiter"]
    lim = VANLEER if lim == HYBRID else lim
    nd, nc, dim, cdim = q.shape[3 - d], q.shape[3 - c], 2 - d, 2 - c
    v = (q[1 + d] / q[0]).index_select(dim, _ghosts(nd, bc, q.device))
    faces = _ghosts(nc, bc, q.device, 1, 1)
    v = v.index_select(cdim, faces)
    Rc, R = _Right(cdim), _Right(dim)
    shape, cshape = [1, 1, 1], [1, 1, 1]
    shape[dim], cshape[cdim] = -1, -1
    wd = None
    if P["widths"] is not None:
        wc = P["widths"][c].index_select(0, faces).view(cshape)
        wd = P["widths"][d].index_select(0, _ghosts(nd, bc, q.device)).view(shape)
        vt = (Rc(wc) * _L(v, Rc) + _L(wc, Rc) * Rc(v)) / (_L(wc, Rc) + Rc(wc))
    else:
        vt = 0.5 * (_L(v, Rc) + Rc(v))
    bf = q[5 + c].index_select(dim, _ghosts(nd, bc, q.device)).index_select(cdim, faces[:-1])
    m = nd + 2 * G
    at = lambda a, k, cnt: a.narrow(dim, k, cnt)  # noqa: E731
    vh = 0.25 * (at(vt, 2, m - 2) + 2.0 * at(vt, 1, m - 2) + at(vt, 0, m - 2))   # cells 1 .. m-2
    bf = at(bf, 1, m - 2)
    w1 = at(wd, 1, m - 2) if wd is not None else None
    if wd is not None:
        vbar = (R(w1) * _L(vh, R) + _L(w1, R) * R(vh)) / (_L(w1, R) + R(w1))
    else:
        vbar = 0.5 * (_L(vh, R) + R(vh))
    w = vh * bf
    f1 = torch.where(vbar > 0, _L(w, R), R(w))
    lam = dt / at(w1, 1, m - 4) if wd is not None else dt / P["h"][d]
    bp = at(bf, 1, m - 4) - 0.5 * lam * (R(f1) - _L(f1, R))                      # cells 2 .. m-3
    wp = at(vh, 1, m - 4) * bp
    k = m - 4                                                                    # cells of wp
    dw = R(wp) - _L(wp, R)
    vb = at(vbar, 2, k - 3)                                                      # interfaces (3,4) ..
    d0, d1, d2 = at(dw, 0, k - 3), at(dw, 1, k - 3), at(dw, 2, k - 3)
    sp = sm = 1.0
    if wd is not None:
        w2 = at(w1, 1, k)
        gap = 0.5 * (_L(w2, R) + R(w2))
        d0, d1, d2 = d0 / at(gap, 0, k - 3), d1 / at(gap, 1, k - 3), d2 / at(gap, 2, k - 3)
        sp, sm = at(w2, 1, k - 3), at(w2, 2, k - 3)
    return torch.where(vb > 0, at(wp, 1, k - 3) + 0.5 * sp * _limit(lim, d0, d1),
                       at(wp, 2, k - 3) - 0.5 * sm * _limit(lim, d1, d2))


def _magnetic(q, d, dt, P):
    dim, out = 2 - d, [None] * 3
    shape = [1, 1, 1]
    shape[dim] = -1
    Rd = _Right(dim)
    bd = q[5 + d]
    for c in ((d + 1) % 3, (d + 2) % 3):
        f = _edge_fluxes(q, d, c, dt, P)
        cshape = [1, 1, 1]
        cshape[2 - c] = -1
        wd = P["widths"][d].view(shape) if P["widths"] is not None else P["h"][d]
        wc = P["widths"][c].view(cshape) if P["widths"] is not None else P["h"][c]
        up = f.narrow(2 - c, 1, f.shape[2 - c] - 1)
        out[c] = q[5 + c] - dt / wd * (Rd(up) - _L(up, Rd))
        right = Rd(f)
        Rc = _Right(2 - c)
        bd = bd + dt / wc * (Rc(right) - _L(right, Rc))
    out[d] = bd
    return torch.cat([q[:5], torch.stack(out)])


def _cfl(q, P):
    b = _centred(q, P["bc"])
    best = None
    for d in range(3):
        v, _, _, _, cf = _speeds(q[0], q[1:4], q[4], b, d, P["gamma"])
        s = v[d].abs() + cf
        if P["widths"] is not None:
            shape = [1, 1, 1]
            shape[2 - d] = -1
            r = float((P["widths"][d].view(shape) / s).min())
        else:
            r = P["h"][d] / float(s.max())
        best = r if best is None else min(best, r)
    return CFL * best


def _advance(q, steps, P):
    dt = None
    for _ in range(steps):
        dt = _cfl(q, P)
        for d, order in ((0, "LB"), (1, "LB"), (2, "LB"), (2, "BL"), (1, "BL"), (0, "BL")):
            for op in order:
                if op == "B":
                    q = _magnetic(q, d, dt, P)
                    continue
                if P["physics"] == "split":
                    q = _kick(q, d, 0.5 * dt, P)
                q = _fluid(q, d, dt, P)
                if P["physics"] == "split":
                    q = _kick(q, d, 0.5 * dt, P)
    return q, dt


def _totals(q, P):
    vol = P["h"][0] * P["h"][1] * P["h"][2]
    return (q.sum(dim=(1, 2, 3)) * vol).cpu().numpy()


def exact(case, seed):
    if _cells(case) > 2.5e7:
        return None
    if case["kind"] == "batch":
        states, dts = [], []
        for w in _batch_boxes(case, seed):
            # the batch holds its boxes in FP32
            q = torch.as_tensor(w.state, device=DEVICE).float().double()
            q, dt = _advance(q, case["steps"], {"gamma": w.gamma, "bc": w.bc, "h": w.h, "limiter": VANLEER,
                                                "physics": "plain", "phi": None, "widths": None})
            states.append(q.cpu().numpy())
            dts.append(dt)
        return {"states": states, "dt": np.array(dts)}
    q, gamma, h, phi, widths = _problem(case, seed)
    P = {"gamma": gamma, "bc": case["bc"], "h": h, "limiter": case["limiter"], "physics": case["physics"],
         "phi": None if phi is None else torch.as_tensor(phi, device=DEVICE),
         "widths": None if widths is None else [torch.as_tensor(x, device=DEVICE) for x in widths]}
    q, dt = _advance(q.double(), case["steps"], P)
    r = {"state": q, "dt": dt}
    if case["monitor"]:
        r["totals"] = _totals(q, P)
    return r
