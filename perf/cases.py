"""The work that a user of this package has it do, as timed cases.

Every case is one call (or the few calls of one step) through the package's
public entry points on inputs made from a seed:

  sweep     one DD sweep: every subdomain's WaveHoltz solve and the transmission
            update (FP32 or FP64, with or without a source, fixed WaveHoltz
            count or a per-subdomain tolerance, Cartesian or curved elements);
            with a source it is the closing sweep of a DD solve, whose
            subdomain solutions are assembled into a global correction
  packed    one sweep of several small problems in one launch (batches, server)
  residual  r = b - K u and its norms on the whole mesh
  solve     a whole solve to a tight tolerance

A sweep in FP32 writes its results into FP64 buffers, but they carry FP32
rounding: a program that keeps such results keeps them in the type that they
were computed in, and so does ``run``.  Whole solves, residuals and FP64 sweeps
are accurate in FP64 and come back as they are.
"""

import math
import random

import numpy as np
import torch

import paper_2606_21695_gb300 as hz

DEV = "cuda"


# ------------------------------------------------------------------ cases --
def _sweep(name, nx, ny, P, sx, sy, omega, speed, **kw):
    c = {"kind": "sweep", "nx": nx, "ny": ny, "P": P, "sx": sx, "sy": sy, "omega": omega, "speed": speed,
         "x0": 0.0, "y0": 0.0, "size": 1.0, "prec": "fp32", "wh": 20, "tol": 0.0, "source": False, "warp": 0.0}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: 16 subdomains of 17 x 17 nodes (the 32 x 32, P = 2 workload)
        _sweep("sweep_p2_16sub", 32, 32, 2, 8, 8, 10.0, "const"),
        # the inner call of the benchmark's solve, about 900 times per solve (256 x 256, P = 3, Y channel)
        _sweep("sweep_p3_1024sub", 256, 256, 3, 8, 8, 64 * math.pi, "channel"),
        # the closing sweep of a DD solve on the same mesh: dense right-hand side in, global correction out
        _sweep("closing_p3_1024sub", 256, 256, 3, 8, 8, 64 * math.pi, "channel", source=True),
        # the largest: the 1024 x 1024, P = 4 random medium, 16.8 M nodes, 129 x 129 nodes a subdomain
        _sweep("sweep_p4_wide", 1024, 1024, 4, 32, 32, 2 * math.pi * 204.8, "random", x0=-1.0, y0=-1.0, size=2.0),
        # an 8 x 8-subdomain piece of it as its solves run it: WaveHoltz to a tolerance per subdomain
        _sweep("sweep_p4_piece_tol", 256, 256, 4, 32, 32, 2 * math.pi * 204.8, "random", x0=-0.5, y0=-0.5, size=0.5,
               wh=60, tol=1e-4),
        # a problem of the batched and served mix: small subdomains of high degree, random medium
        _sweep("sweep_p5_small", 128, 128, 5, 4, 4, 80.0, "random", wh=5),
        # subdomain shape with no power of two in it, non-square mesh
        _sweep("sweep_p3_ragged", 96, 60, 3, 12, 10, 60.0, "channel", wh=10),
        # the plain FP64 path, a quarter of the benchmark's mesh at its own resolution
        _sweep("sweep64_p3_256sub", 128, 128, 3, 8, 8, 64 * math.pi, "channel", x0=0.25, y0=0.25, size=0.5,
               prec="fp64", wh=10),
        # curved quadrilaterals: the benchmark's mesh with warped elements
        _sweep("sweep_curved_p3", 256, 256, 3, 8, 8, 64 * math.pi, "channel", warp=0.03, wh=10),
        # the residual that every refinement and every FGMRES step computes, on the benchmark's mesh
        {"name": "residual_p3", "kind": "residual", "nx": 256, "ny": 256, "P": 3, "sx": 8, "sy": 8,
         "omega": 64 * math.pi, "speed": "channel", "x0": 0.0, "y0": 0.0, "size": 1.0},
        # batches and the server: the sweeps of problems of several degrees and sizes in one launch
        {"name": "packed_12", "kind": "packed", "problems": 12, "mix": 4, "wh": 5},
        # a whole solve (FP32 sweeps inside FP64 flexible GMRES) as the benchmark runs it, a quarter of its mesh
        {"name": "solve_p3_256sub", "kind": "solve", "nx": 128, "ny": 128, "P": 3, "sx": 8, "sy": 8,
         "omega": 64 * math.pi, "speed": "channel", "x0": 0.25, "y0": 0.25, "size": 0.5, "prec": "fp32", "tol": 1e-12},
    ]


MAX_UPDATES = 1.5e10  # DOF-updates of the largest listed sweep


def _updates(c):
    return (c["nx"] // c["sx"]) * (c["ny"] // c["sy"]) * (c["sx"] * c["P"] + 1) * (c["sy"] * c["P"] + 1) * c["wh"]


def draw(rng):
    kind = rng.choices(["sweep", "residual", "packed", "solve"], [14, 2, 2, 1])[0]
    if kind == "packed":
        return {"kind": "packed", "problems": rng.randint(3, 24), "mix": rng.randint(5, 10**6), "wh": rng.choice([3, 5, 10])}
    if kind == "residual":
        P = rng.choice([1, 2, 3, 4, 5, 7])
        nx = int(round(math.exp(rng.uniform(math.log(24), math.log(3000 / P)))))
        ny = int(round(math.exp(rng.uniform(math.log(24), math.log(3000 / P)))))
        return {"kind": "residual", "nx": nx, "ny": ny, "P": P, "sx": nx, "sy": ny, "omega": rng.uniform(5.0, 200.0),
                "speed": rng.choice(["channel", "random"]), "x0": 0.0, "y0": 0.0, "size": 1.0}
    if kind == "solve":
        n = rng.choice([32, 40, 48, 64])
        return {"kind": "solve", "nx": n, "ny": n, "P": rng.choice([2, 3]), "sx": 8, "sy": 8, "omega": rng.uniform(40.0, 80.0),
                "speed": rng.choice(["const", "channel"]), "x0": 0.0, "y0": 0.0, "size": 1.0, "prec": "fp32", "tol": 1e-12}
    while True:
        what = rng.choices(["plain", "source", "tol", "fp64", "curved"], [7, 2, 2, 2, 1])[0]
        P = rng.choice([2, 3, 4, 5]) if rng.random() < 0.85 else rng.choice([1, 6, 7])
        s = rng.choice([4, 8, 16, 32])  # subdomains of the batched workload's sampler, some of them ragged
        sx, sy = (s, s) if rng.random() < 0.7 else (rng.choice([3, 4, 5, 6, 8, 10, 12, 16]), rng.choice([3, 4, 6, 7, 8, 12, 16]))
        if P >= 5 and max(sx, sy) > (16, 8)[P > 5]:
            continue  # wider than any subdomain in use
        if what == "curved" and (sx * P + 1) * (sy * P + 1) > 1024:
            continue
        S = math.exp(rng.uniform(math.log(4), math.log(1024 if s < 32 else 256)))
        Sx = max(1, int(round(math.sqrt(S) * rng.uniform(0.7, 1.4))))
        Sy = max(1, int(round(S / Sx)))
        nx, ny = Sx * sx, Sy * sy
        # 8 to 40 node spacings per wavelength at c = 1
        omega = 2 * math.pi * max(nx, ny) * P / math.exp(rng.uniform(math.log(8), math.log(40)))
        c = _sweep(None, nx, ny, P, sx, sy, omega, rng.choice(["channel", "random"]) if what != "curved" else "channel",
                   wh=rng.choice([3, 5, 10, 20]))
        if what == "source":
            c["source"] = True
        elif what == "tol":
            c.update(wh=40, tol=1e-4)
        elif what == "fp64":
            c["prec"] = "fp64"
        elif what == "curved":
            c["warp"] = rng.uniform(0.01, 0.04)
        cost = _updates(c) * _nt(c) * (1, 30)[c["prec"] == "fp64"] * (1, 4)[c["warp"] > 0]
        if cost <= MAX_UPDATES and c["wh"] * _nt(c) <= 4000:
            return c


# ----------------------------------------------- spectral elements (FP64) --
def _gll(P):
    """GLL nodes, weights and differentiation matrix D[q, a] = l_a'(x_q) on [-1, 1]."""
    L = np.polynomial.legendre.Legendre.basis(P)
    x = np.concatenate([[-1.0], np.sort(L.deriv().roots().real) if P > 1 else [], [1.0]])
    for _ in range(3):  # polish the interior roots
        if P > 1:
            x[1:-1] -= L.deriv()(x[1:-1]) / L.deriv(2)(x[1:-1])
    w = 2.0 / (P * (P + 1) * L(x) ** 2)
    D = np.zeros((P + 1, P + 1))
    for q in range(P + 1):
        for a in range(P + 1):
            if q != a:
                D[q, a] = L(x[q]) / (L(x[a]) * (x[q] - x[a]))
    D[0, 0], D[P, P] = -P * (P + 1) / 4.0, P * (P + 1) / 4.0
    return x, w, D


def _assemble_1d(n, P, h):
    """Assembled stiffness (n P + 1)^2 and lumped weights of n elements of length h."""
    _, w, D = _gll(P)
    Kr = D.T @ np.diag(w) @ D
    N = n * P + 1
    K, W = np.zeros((N, N)), np.zeros(N)
    for e in range(n):
        i = e * P
        K[i:i + P + 1, i:i + P + 1] += 2.0 / h * Kr
        W[i:i + P + 1] += w * h / 2.0
    return K, W


def _coords(n, P, x0, h):
    x, _, _ = _gll(P)
    g = x0 + (np.arange(n)[:, None] + (x[None, :P] + 1.0) / 2.0) * h
    return np.concatenate([g.ravel(), [x0 + n * h]])


def _steps(c):
    return c["size"] / c["nx"], c["size"] / c["ny"]


def _max_eig(n, P, h):
    K, W = _assemble_1d(n, P, h)
    s = 1.0 / np.sqrt(W)
    return float(np.linalg.eigvalsh(K * s[:, None] * s[None, :])[-1])


def _nt(c):
    """Time steps per period at 0.9 of the leapfrog limit for the largest wave speed of the medium (1.75 or 1)."""
    hx, hy = _steps(c)
    cmax = 1.75 if c["speed"] == "random" else 1.0
    lam = cmax**2 * (_max_eig(min(c["sx"], 8), c["P"], hx) + _max_eig(min(c["sy"], 8), c["P"], hy)) * 1.02
    margin = 1.35 if c.get("warp", 0.0) > 0 else 1.0  # curved elements are up to a third narrower
    return max(3, math.ceil(2 * math.pi / c["omega"] / (0.9 * 2.0 / math.sqrt(lam)) * margin))


# ------------------------------------------------------------------ inputs --
def _segment_distance(X, Y, a, b):
    dx, dy = b[0] - a[0], b[1] - a[1]
    t = (((X - a[0]) * dx + (Y - a[1]) * dy) / (dx * dx + dy * dy)).clamp(0.0, 1.0)
    return torch.hypot(X - (a[0] + t * dx), Y - (a[1] + t * dy))


def _speed(c, X, Y, rng):
    """Nodal wave speed at X, Y (NY, NX): 1, a Y-shaped channel at 1/3, or a smooth random medium in [0.25, 1.75]."""
    if c["speed"] == "const":
        return torch.ones_like(X)
    if c["speed"] == "channel":
        shift = rng.uniform(-0.02, 0.02)
        d = None
        for a, b in (((0.5, 0.0), (0.5, 0.5)), ((0.5, 0.5), (0.2, 1.0)), ((0.5, 0.5), (0.8, 1.0))):
            q = _segment_distance(X - shift, Y, a, b)
            d = q if d is None else torch.minimum(d, q)
        return torch.where(d <= 0.04, 1.0 / 3.0, 1.0).double()
    g = np.random.default_rng(rng.randrange(1 << 30))
    kx, ky = g.standard_normal(256) / 0.05, g.standard_normal(256) / 0.05
    ph = g.uniform(0.0, 2 * math.pi, 256)
    kx, ky, ph = (torch.from_numpy(v).to(X.device) for v in (kx, ky, ph))
    ax, ay = X[0][None, :] * kx[:, None] + ph[:, None], Y[:, 0][:, None] * ky[None, :]
    f = math.sqrt(2.0 / 256) * (torch.cos(ay) @ torch.cos(ax) - torch.sin(ay) @ torch.sin(ax))
    return 1.0 + 0.5 * f.clamp(-1.5, 1.5)


def _fields(c, seed):
    """Node positions, wave speed, source and random draws of one case, on the GPU in FP64."""
    rng = random.Random(seed * 7919 + 17)
    hx, hy = _steps(c)
    gx = torch.from_numpy(_coords(c["nx"], c["P"], c["x0"], hx)).to(DEV)
    gy = torch.from_numpy(_coords(c["ny"], c["P"], c["y0"], hy)).to(DEV)
    Y, X = torch.meshgrid(gy, gx, indexing="ij")
    if c.get("warp", 0.0) > 0:
        s, t = (X - c["x0"]) / c["size"], (Y - c["y0"]) / c["size"]
        X, Y = (X + c["warp"] * c["size"] * torch.sin(2 * math.pi * s) * torch.sin(math.pi * t),
                Y + c["warp"] * c["size"] * torch.sin(math.pi * s) * torch.sin(2 * math.pi * t))
    speed = _speed(c, X, Y, rng)
    gen = torch.Generator(device=DEV).manual_seed(rng.randrange(1 << 30))
    sx, sy = (c["x0"] + c["size"] * rng.uniform(0.3, 0.7) for _ in range(2))
    sy += c["y0"] - c["x0"]
    width = max(0.25 * 2 * math.pi * float(speed.min()) / c["omega"], 2.0 * max(hx, hy) / c["P"])
    src = torch.exp(-((X - sx) ** 2 + (Y - sy) ** 2) / (2 * width**2)) / (2 * math.pi * width**2)
    return {"X": X, "Y": Y, "c": speed, "f": src.to(torch.complex128), "gen": gen}


def _randn(shape, gen):
    return torch.view_as_complex(torch.randn(*shape, 2, dtype=torch.float64, device=DEV, generator=gen))


def _lam_in(c, gen):
    """Incoming transmission data: complex normal on every interface, zero on the outer boundary and in the padding."""
    Sx, Sy = c["nx"] // c["sx"], c["ny"] // c["sy"]
    nlx, nly = c["sx"] * c["P"] + 1, c["sy"] * c["P"] + 1
    lam = _randn((Sy, Sx, 4, max(nlx, nly)), gen)
    lam[:, :, 0:2, nly:] = 0
    lam[:, :, 2:4, nlx:] = 0
    lam[:, 0, 0] = 0
    lam[:, -1, 1] = 0
    lam[0, :, 2] = 0
    lam[-1, :, 3] = 0
    return lam


class _State:
    """A mesh, a problem and a user's device buffers."""

    def __init__(self, c, seed):
        self.case = c
        self.fields = f = _fields(c, seed)
        self.mesh = hz.hz_mesh_create(c["x0"], c["x0"] + c["size"], c["y0"], c["y0"] + c["size"], c["nx"], c["ny"],
                                      c["P"], c["sx"], c["sy"])
        self.pr = hz.hz_problem_create(self.mesh, 0)
        self.n = n = hz.hz_mesh_num_nodes(self.mesh)
        if c.get("warp", 0.0) > 0:
            hz.hz_problem_set(self.pr, hz.HZ_NODE_COORDS, torch.stack([f["X"], f["Y"]], -1).cpu().numpy())
        hz.hz_problem_set_device(self.pr, hz.HZ_WAVE_SPEED, f["c"].contiguous(), n)
        hz.hz_problem_set_device(self.pr, hz.HZ_SOURCE, f["f"].contiguous(), n)
        hz.hz_problem_set(self.pr, hz.HZ_OMEGA, np.array([c["omega"]]))

    def __del__(self):
        try:
            hz.hz_problem_destroy(self.pr)
            hz.hz_mesh_destroy(self.mesh)
        except Exception:
            pass


PRECISION = {"fp32": hz.HZ_FP32_REFINE, "fp64": hz.HZ_FP64}


def _sweep_state(c, seed):
    s = _State(c, seed)
    gen = s.fields["gen"]
    L = (c["nx"] // c["sx"]) * (c["ny"] // c["sy"])
    s.nt = _nt(c)
    hz.hz_prepare(s.pr, s.nt)
    s.lam_in = _lam_in(c, gen)
    s.lam_out = torch.zeros_like(s.lam_in)
    s.rhs = None
    s.u_sub = torch.zeros((L, c["sy"] * c["P"] + 1, c["sx"] * c["P"] + 1), dtype=torch.complex128, device=DEV)
    if c.get("source"):
        s.rhs = _randn(tuple(s.fields["X"].shape), gen) * (s.fields["X"].numel() ** -0.5)
        s.u = torch.zeros_like(s.rhs)
    s.fields = None
    return s


def _packed_cases(c):
    """Small problems of the degrees and shapes that the packed launch takes."""
    rng = random.Random(c["mix"])
    out = []
    for _ in range(c["problems"]):
        P, s = rng.choice([(1, 8), (2, 4), (2, 8), (3, 4), (3, 8), (4, 4), (5, 4)])
        S = rng.choice([2, 3, 4, 6, 8])
        n = s * S
        omega = 2 * math.pi * n * P / math.exp(rng.uniform(math.log(8), math.log(30)))
        out.append(_sweep(None, n, n, P, s, s, omega, rng.choice(["channel", "random"]), wh=c["wh"]))
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        return _sweep_state(case, seed)
    if kind == "packed":
        return [_sweep_state(c, seed * 100 + k) for k, c in enumerate(_packed_cases(case))]
    s = _State(case, seed)
    shape = tuple(s.fields["X"].shape)
    if kind == "residual":
        gen = s.fields["gen"]
        s.b, s.u = _randn(shape, gen), _randn(shape, gen)
        s.r, s.norms = torch.zeros_like(s.u), torch.zeros(2, dtype=torch.float64, device=DEV)
    else:
        s.u = torch.zeros(shape, dtype=torch.complex128, device=DEV)
        # the benchmark's outer iteration: DD solves to 0.3 inside FGMRES(60)
        s.opts = hz.hz_default_opts(precision=PRECISION[case["prec"]], tol=case["tol"], refine=hz.HZ_REFINE_FGMRES,
                                    refine_restart=60, inner_tol=0.3, max_refine=200, max_sweeps=20000)
    s.fields = None
    return s


def _as_computed(t, prec):
    return torch.view_as_real(t).to(torch.float32) if prec == "fp32" else torch.view_as_real(t)


def run(state):
    if isinstance(state, list):
        wh = state[0].case["wh"]
        hz.hz_sweep_packed([s.pr for s in state], [s.nt for s in state], wh, [s.lam_in for s in state],
                           [s.lam_out for s in state], None, [s.u_sub for s in state])
        return [[_as_computed(s.lam_out, "fp32"), _as_computed(s.u_sub, "fp32")] for s in state]
    c = state.case
    if c["kind"] == "residual":
        hz.hz_residual(state.pr, state.b, state.u, state.r, state.norms)
        return [state.r, state.norms]
    if c["kind"] == "solve":
        hz.hz_solve_device(state.pr, state.opts, state.u)
        return [state.u]
    hz.hz_sweep(state.pr, PRECISION[c["prec"]], state.nt, c["wh"], c["tol"], state.lam_in, state.lam_out, state.rhs,
                state.u_sub)
    out = [_as_computed(state.lam_out, c["prec"])]
    if c["source"]:
        state.u.zero_()
        hz.hz_assemble_add(state.pr, state.u_sub, state.u)
        out.append(_as_computed(state.u, c["prec"]))
    else:
        out.append(_as_computed(state.u_sub, c["prec"]))
    return out


# -------------------------------------------------------------------- work --
def _sweep_work(c):
    """Each input read once, each output written once; per node and time step the leapfrog update, the two filter
    sums and the banded (or, on curved elements, the element-wise) stiffness apply."""
    P, nt = c["P"], _nt(c)
    nlx, nly = c["sx"] * P + 1, c["sy"] * P + 1
    L = (c["nx"] // c["sx"]) * (c["ny"] // c["sy"])
    nodes = L * nlx * nly
    lam = 2 * 16 * 4 * L * max(nlx, nly)
    real = 4 if c["prec"] == "fp32" else 8
    n = (c["nx"] * P + 1) * (c["ny"] * P + 1)
    out = 16 * n * 2 if c["source"] else 16 * nodes
    if c["warp"] > 0:
        en = c["sx"] * c["sy"] * (P + 1) ** 2 * L
        fma = en * (4 * (P + 1) + 4) + nodes * 7
        data = en * 3 * real + nodes * real
    else:
        taps = 2 * ((2 * P + 1) + (P - 1) * (P + 1)) / P  # x and y, averaged over the nodes of an element
        fma = nodes * (taps + 5)
        data = nodes * real
    return {"bytes": lam + data + out, "flops": 2.0 * fma * (nt - 1) * c["wh"]}


def work(case):
    if case["kind"] == "sweep":
        w = _sweep_work(case)
        if case["tol"] > 0:  # about half of the allowed WaveHoltz iterations
            w["flops"] *= 0.5
        return w
    if case["kind"] == "packed":
        ws = [_sweep_work(c) for c in _packed_cases(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    P = case["P"]
    n = (case["nx"] * P + 1) * (case["ny"] * P + 1)
    taps = 2 * ((2 * P + 1) + (P - 1) * (P + 1)) / P
    if case["kind"] == "residual":
        return {"bytes": 56 * n, "flops": n * (4 * taps + 16)}
    # a solve: about 0.5 sweeps of 20 WaveHoltz iterations per subdomain row and decade of the residual
    sweeps = 6 * math.sqrt(n) / (case["sx"] * P) * 2
    one = _sweep_work(_sweep(None, case["nx"], case["ny"], P, case["sx"], case["sy"], case["omega"], case["speed"],
                             size=case["size"]))
    return {"bytes": 16 * n * 3, "flops": one["flops"] * sweeps}


# ------------------------------------------------------------------- exact --
def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _split(c, full):
    """Global nodes (NY, NX) as subdomain copies (L, nly, nlx)."""
    a, b = c["sx"] * c["P"], c["sy"] * c["P"]
    s = full.unfold(0, b + 1, b).unfold(1, a + 1, a)
    return s.reshape(-1, b + 1, a + 1)


def _curved_geometry(c, f):
    """Per element node: metric (G11, G12, G22) and lumped weight; lumped weights on the subdomains, their share of the
    global ones and the arc-length edge weights (L, 4, NE)."""
    P, M = c["P"], c["P"] + 1
    _, w, D = _gll(P)
    D, w = _t(D), _t(w)

    def elements(z):  # (L, sy, sx, M, M)
        s = _split(c, z)
        return s.unfold(1, M, P).unfold(2, M, P)

    X, Y = elements(f["X"]), elements(f["Y"])
    xx, yx = X @ D.T, Y @ D.T
    xe, ye = D @ X, D @ Y
    J = xx * ye - xe * yx
    ww = w[:, None] * w[None, :]
    G = (ww * (xe**2 + ye**2) / J, -ww * (xx * xe + yx * ye) / J, ww * (xx**2 + yx**2) / J)
    return D, w, G, ww * J, torch.sqrt(xx**2 + yx**2), torch.sqrt(xe**2 + ye**2)


def _gather(c, E):
    """Sum of element values (L, sy, sx, M, M) at the subdomain nodes (L, nly, nlx)."""
    P, M = c["P"], c["P"] + 1
    L = E.shape[0]
    out = torch.zeros(L, c["sy"] * P + 1, c["sx"] * P + 1, dtype=E.dtype, device=E.device)
    for b in range(M):
        for a in range(M):
            out[:, b:b + P * (c["sy"] - 1) + 1:P, a:a + P * (c["sx"] - 1) + 1:P] += E[:, :, :, b, a]
    return out


def _exact_sweep(c, seed):
    """The sweep's definition in FP64: WaveHoltz with the modified leapfrog on every subdomain, then
    lambda_out = -lambda_in - 2 i k u at the neighbour's side of each interface."""
    f = _fields(c, seed)
    P, nt, w = c["P"], _nt(c), c["omega"]
    Sx, Sy = c["nx"] // c["sx"], c["ny"] // c["sy"]
    L, nlx, nly = Sx * Sy, c["sx"] * P + 1, c["sy"] * P + 1
    hx, hy = _steps(c)
    lam = _lam_in(c, f["gen"])
    rhs = _randn(tuple(f["X"].shape), f["gen"]) * (f["X"].numel() ** -0.5) if c["source"] else None
    cs = _split(c, f["c"])
    Kx, Wx = _assemble_1d(c["sx"], P, hx)
    Ky, Wy = _assemble_1d(c["sy"], P, hy)
    Kx, Wx, Ky, Wy = (_t(v) for v in (Kx, Wx, Ky, Wy))
    if c["warp"] > 0:
        D, w1, G, JW, sxi, seta = _curved_geometry(c, f)
        W = _gather(c, JW)
        edge = torch.zeros(L, 4, max(nlx, nly), dtype=torch.float64, device=DEV)
        for e in range(c["sy"]):
            edge[:, 0, e * P:e * P + P + 1] += w1 * seta[:, e, 0, :, 0]
            edge[:, 1, e * P:e * P + P + 1] += w1 * seta[:, e, -1, :, P]
        for e in range(c["sx"]):
            edge[:, 2, e * P:e * P + P + 1] += w1 * sxi[:, 0, e, 0, :]
            edge[:, 3, e * P:e * P + P + 1] += w1 * sxi[:, -1, e, P, :]

        def stiff(p):
            u = p.unfold(1, P + 1, P).unfold(2, P + 1, P)
            ux, ue = u @ D.T, D @ u
            return _gather(c, (G[0] * ux + G[1] * ue) @ D + D.T @ (G[1] * ux + G[2] * ue))
    else:
        W = Wy[:, None] * Wx[None, :] * torch.ones_like(cs)
        edge = torch.zeros(L, 4, max(nlx, nly), dtype=torch.float64, device=DEV)
        edge[:, 0:2, :nly] = Wy
        edge[:, 2:4, :nlx] = Wx

        def stiff(p):
            return Wy[:, None] * (p @ Kx) + Wx[None, :] * (Ky @ p)
    b = torch.zeros_like(cs, dtype=torch.complex128)
    if rhs is not None:
        ones = torch.ones_like(f["X"])
        if c["warp"] > 0:
            raise ValueError("no curved case has a source")
        cover = torch.zeros_like(ones)  # subdomains that share a node
        a_, b_ = c["sx"] * P, c["sy"] * P
        for sy in range(Sy):
            for sx in range(Sx):
                cover[sy * b_:sy * b_ + b_ + 1, sx * a_:sx * a_ + a_ + 1] += 1
        b += _split(c, rhs / cover)
    lam4 = lam.reshape(L, 4, -1)
    b[:, :, 0] += edge[:, 0, :nly] * lam4[:, 0, :nly]
    b[:, :, -1] += edge[:, 1, :nly] * lam4[:, 1, :nly]
    b[:, 0, :] += edge[:, 2, :nlx] * lam4[:, 2, :nlx]
    b[:, -1, :] += edge[:, 3, :nlx] * lam4[:, 3, :nlx]
    H = torch.zeros_like(cs)
    H[:, :, 0] += edge[:, 0, :nly]
    H[:, :, -1] += edge[:, 1, :nly]
    H[:, 0, :] += edge[:, 2, :nlx]
    H[:, -1, :] += edge[:, 3, :nlx]
    H, M = H / cs, W / cs**2
    dt = 2 * math.pi / w / nt
    theta, sigma = math.tan(w * dt / 2) / w, math.sin(w * dt / 2) / (w / 2)
    alpha, beta = (M - theta * H) / (M + theta * H), sigma / (M + theta * H)
    br, bi = (beta * b.real).contiguous(), (beta * b.imag).contiguous()
    c0 = -0.25 + 0.25 * math.tan(math.pi / nt) ** 2
    u = torch.zeros_like(b)
    live = torch.ones(L, dtype=torch.bool, device=DEV)
    for _ in range(c["wh"]):
        p = u.real.contiguous()
        pd = w * (u.imag * math.cos(math.pi / nt) - u.real * math.sin(math.pi / nt))
        vr, vi = (1 + c0) * p, (math.cos(math.pi / nt) + c0) / w * pd
        for nu in range(1, nt):
            th = 2 * math.pi * nu / nt
            p = p + sigma * pd
            pd = alpha * pd - beta * stiff(p) + math.cos(th) * br + math.sin(th) * bi
            vr += (math.cos(th) + c0) * p
            vi += (math.cos(2 * math.pi * (nu + 0.5) / nt) + c0) / w * pd
        new = torch.complex(vr, vi) * (2.0 / nt)
        if c["tol"] > 0:
            new = torch.where(live[:, None, None], new, u)
            d, q = ((new - u).abs() ** 2).sum((1, 2)), (new.abs() ** 2).sum((1, 2))
            live &= ~(d <= c["tol"] ** 2 * q)
        u = new
        if not bool(live.any()):
            break
    k = w / cs
    out = torch.zeros_like(lam)
    g4, k4 = u.reshape(Sy, Sx, nly, nlx), k.reshape(Sy, Sx, nly, nlx)
    out[:, 1:, 0, :nly] = (-lam[:, :-1, 1, :nly] - 2j * k4[:, :-1, :, -1] * g4[:, :-1, :, -1])
    out[:, :-1, 1, :nly] = (-lam[:, 1:, 0, :nly] - 2j * k4[:, 1:, :, 0] * g4[:, 1:, :, 0])
    out[1:, :, 2, :nlx] = (-lam[:-1, :, 3, :nlx] - 2j * k4[:-1, :, -1, :] * g4[:-1, :, -1, :])
    out[:-1, :, 3, :nlx] = (-lam[1:, :, 2, :nlx] - 2j * k4[1:, :, 0, :] * g4[1:, :, 0, :])
    if not c["source"]:
        return [torch.view_as_real(out), torch.view_as_real(u)]
    full = torch.zeros_like(rhs)
    for sy in range(Sy):
        for sx in range(Sx):
            full[sy * b_:sy * b_ + b_ + 1, sx * a_:sx * a_ + a_ + 1] += g4[sy, sx]
    return [torch.view_as_real(out), torch.view_as_real(full / cover)]


def _operator(c, f):
    """Assembled 1D factors and the diagonal of K = A - i w H - w^2 M on the whole mesh."""
    hx, hy = _steps(c)
    Kx, Wx = (_t(v) for v in _assemble_1d(c["nx"], c["P"], hx))
    Ky, Wy = (_t(v) for v in _assemble_1d(c["ny"], c["P"], hy))
    H = torch.zeros_like(f["c"])
    H[0, :] += Wx
    H[-1, :] += Wx
    H[:, 0] += Wy
    H[:, -1] += Wy
    w = c["omega"]
    diag = torch.complex(-w * w * Wy[:, None] * Wx[None, :] / f["c"] ** 2, -w * H / f["c"])
    return Kx, Wx, Ky, Wy, diag


def _exact_residual(c, seed):
    f = _fields(c, seed)
    shape = tuple(f["X"].shape)
    b, u = _randn(shape, f["gen"]), _randn(shape, f["gen"])
    Kx, Wx, Ky, Wy, diag = _operator(c, f)

    def A(v):
        return Wy[:, None] * (v @ Kx) + Wx[None, :] * (Ky @ v)

    r = b - torch.complex(A(u.real.contiguous()), A(u.imag.contiguous())) - diag * u
    return [r, torch.stack([(r.abs() ** 2).sum(), (b.abs() ** 2).sum()])]


def _exact_solve(c, seed):
    """Direct solve of K u = b: block elimination over element rows."""
    f = _fields(c, seed)
    Kx, Wx, Ky, Wy, diag = _operator(c, f)
    P, NX, NY = c["P"], Wx.numel(), Wy.numel()
    b = Wy[:, None] * Wx[None, :] * f["f"]
    Dx = torch.diag(Wx)

    def block(rows, cols):
        K = torch.kron(Ky[rows][:, cols].contiguous(), Dx).to(torch.complex128)
        if rows == cols:
            K += torch.kron(torch.diag(Wy[rows]), Kx)
            K += torch.diag(diag[rows].reshape(-1))
        return K

    groups = [slice(j, min(j + P, NY)) for j in range(0, NY, P)]
    lu = []
    for i, g in enumerate(groups):
        S, y = block(g, g), b[g].reshape(-1, 1)
        if i:
            low = block(g, groups[i - 1])
            S = S - low @ lu[-1][1]
            y = y - low @ lu[-1][2]
        F = torch.linalg.lu_factor(S)
        up = block(g, groups[i + 1]) if i + 1 < len(groups) else None
        Z = None
        if up is not None:
            Z = torch.zeros_like(up)  # only the next group's first row is coupled
            Z[:, :NX] = torch.linalg.lu_solve(*F, up[:, :NX].contiguous())
        lu.append((F, Z, torch.linalg.lu_solve(*F, y)))
    x, out = None, []
    for F, Z, y in reversed(lu):
        x = y if Z is None else y - Z @ x
        out.append(x.reshape(-1, NX))
    return [torch.cat(out[::-1], 0)]


def exact(case, seed):
    if case["kind"] == "sweep":
        return _exact_sweep(case, seed)
    if case["kind"] == "packed":
        return [_exact_sweep(c, seed * 100 + k) for k, c in enumerate(_packed_cases(case))]
    if case["kind"] == "residual":
        return _exact_residual(case, seed)
    return _exact_solve(case, seed)
