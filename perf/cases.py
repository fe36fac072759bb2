"""The work the solver is measured on: whole passes through the public calls of
paper_1710_09995_gb300.gbcfd, with inputs made from a seed.

A pass of a flow case hands the solver a conserved state on the GPU (as a run that starts or
restarts, an ensemble member or a service's request does), advances it some time steps and reads
the state back; the steady channel also reads its residual norm, as a convergence loop does.  A
pass of the learned accelerator is one forward pass over a block's features, or one training step.

Sizes are those of the repository's configurations, tests and benchmark: the 32^3 Gaussian pulse,
the 256^3 vortex, lattices of uneven blocks with sides 16..160, the warped grid, the 192x96x64
bump channel and the 192x96x4 slices the accelerator is trained on.

exact() restates the schemes in plain torch float64 (nothing of this repository's solver in it).
"""
import math

import numpy as np
import torch

from paper_1710_09995_gb300 import gbcfd

GAMMA, PRANDTL, EPS = 1.4, 0.72, 0.1
WCNS_EPS = 1e-6
LR = 2e-3
CHANNELS = (10, 32, 32, 5)
F64 = torch.float64


# ---- the cases ------------------------------------------------------------------------------------

def _flow(kind, nx, ny, nz, precision, steps, viscous, limiter=0):
    return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "precision": precision, "steps": steps,
            "viscous": viscous, "limiter": limiter}


def _lattice(bx, by, bz, lo, hi, sizes_seed, precision, steps):
    return {"kind": "lattice", "bx": bx, "by": by, "bz": bz, "lo": lo, "hi": hi, "sizes_seed": sizes_seed,
            "precision": precision, "steps": steps}


def listed():
    return [
        # the smallest runs: a 32^3 Euler block for ten steps, where launches and tails count
        dict(_flow("block", 32, 32, 32, "fp64", 10, False), name="pulse_32_fp64"),
        # a single large Navier-Stokes block in the paper's precision: one step of a long march
        dict(_flow("block", 256, 256, 256, "fp64", 1, True), name="vortex_256_fp64"),
        # the same block in mixed precision (FP32 fluxes, FP64 state), four steps
        dict(_flow("block", 256, 256, 256, "mixed", 4, True), name="vortex_256_mixed"),
        # a multi-zone grid of uneven blocks advanced as one group, FP64 Euler
        dict(_lattice(3, 3, 4, 16, 96, 4, "fp64", 1), name="lattice_36_fp64"),
        # a larger one in mixed precision
        dict(_lattice(3, 3, 4, 16, 160, 4, "mixed", 2), name="lattice_36_mixed"),
        # a curvilinear Navier-Stokes block (the warped periodic grid), mixed precision
        dict(_flow("warped", 256, 256, 192, "mixed", 2, True), name="warped_256_mixed"),
        # the steady bump channel's iteration (walls, far field, local time steps), FP64: the
        # finish of a hybrid solve and the plain iteration
        dict(_flow("channel", 192, 96, 64, "fp64", 2, False), name="channel_fp64"),
        # the same iteration in mixed precision: most of a hybrid solve
        dict(_flow("channel", 192, 96, 64, "mixed", 20, False), name="channel_mixed"),
        # the paper's own scheme (WCNS-E-5, fourth-order viscous terms), FP64
        dict(_flow("wcns", 128, 128, 128, "fp64", 1, True), name="wcns_128_fp64"),
        # the same at the benchmark's size in mixed precision
        dict(_flow("wcns", 256, 256, 256, "mixed", 1, True), name="wcns_256_mixed"),
        # one prediction of the accelerator over the channel's block
        {"kind": "accel_forward", "nx": 192, "ny": 96, "nz": 64, "batch": 1, "name": "accel_forward"},
        # one training step of the accelerator on a batch of four channel slices
        {"kind": "accel_train", "nx": 192, "ny": 96, "nz": 4, "batch": 4, "name": "accel_train"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sides(rng, lo, hi, most):
    while True:
        n = [_log_int(rng, lo, hi) for _ in range(3)]
        if n[0] * n[1] * n[2] <= most:
            return n


def draw(rng):
    kind = rng.choice(["block", "block", "block", "lattice", "lattice", "warped", "channel", "wcns", "wcns",
                       "accel_forward", "accel_train"])
    if kind == "accel_forward":
        nx, ny, nz = _sides(rng, 16, 256, 2_000_000)
        return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "batch": 1}
    if kind == "accel_train":
        return {"kind": kind, "nx": _log_int(rng, 48, 200), "ny": _log_int(rng, 24, 100), "nz": rng.randint(2, 5),
                "batch": rng.randint(1, 4)}
    precision = rng.choice(["fp64", "mixed"])
    if kind == "lattice":
        bx, by, bz = (rng.randint(2, 4) for _ in range(3))
        while bx * by * bz > 36:
            bx, by, bz = (rng.randint(2, 4) for _ in range(3))
        hi = rng.randint(32, 64) if precision == "fp64" else rng.randint(48, 120)
        return _lattice(bx, by, bz, 16, hi, rng.randint(0, 1000), precision, 1 if precision == "fp64" else rng.randint(1, 4))
    most = {("block", "fp64"): 6_000_000, ("block", "mixed"): 12_000_000, ("wcns", "fp64"): 2_000_000,
            ("wcns", "mixed"): 8_000_000, ("warped", "fp64"): 2_000_000, ("warped", "mixed"): 8_000_000,
            ("channel", "fp64"): 2_000_000, ("channel", "mixed"): 4_000_000}[(kind, precision)]
    steps = rng.randint(1, 4)
    nx, ny, nz = _sides(rng, 16, 256, most // steps)
    viscous = kind != "channel" and rng.random() < 0.6
    limiter = 1 if rng.random() < 0.2 else 0
    return _flow(kind, nx, ny, nz, precision, steps, viscous, limiter)


# ---- inputs ----------------------------------------------------------------------------------------

def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _slab_sizes(case):
    rng = np.random.Generator(np.random.PCG64(case["sizes_seed"]))
    return [rng.integers(case["lo"], case["hi"] + 1, size=case[k]).tolist() for k in ("bx", "by", "bz")]


def _extent(case):
    if case["kind"] == "lattice":
        return tuple(sum(s) for s in _slab_sizes(case))
    return case["nx"], case["ny"], case["nz"]


def _conserved(r, u, v, w, p):
    q = torch.empty((5,) + tuple(r.shape), dtype=F64, device=r.device)
    q[0] = r
    q[1] = r * u
    q[2] = r * v
    q[3] = r * w
    q[4] = p / (GAMMA - 1.0) + 0.5 * r * (u * u + v * v + w * w)
    return q


def _waves(shape, rng, amp, dev, modes=3):
    """a seeded sum of periodic Fourier modes (|k| <= 3 per direction), at most `amp` in magnitude"""
    nx, ny, nz = shape
    s = [(torch.arange(n, dtype=F64, device=dev) + 0.5) / n for n in (nx, ny, nz)]
    out = torch.zeros((nz, ny, nx), dtype=F64, device=dev)
    for _ in range(modes):
        k, ph = rng.integers(1, 4, size=3) * rng.choice([-1, 1], size=3), rng.random(3) * 2.0 * math.pi
        f = [torch.sin(2.0 * math.pi * int(k[d]) * s[d] + float(ph[d])) for d in range(3)]
        out += f[2][:, None, None] * f[1][None, :, None] * f[0][None, None, :] * (amp / modes * float(rng.uniform(0.5, 1.0)))
    return out


def _vortex(shape, rng, dev):
    """an isentropic vortex of seeded strength and place in a Mach 0.5 stream on a 10 x 10 box"""
    nx, ny, nz = shape
    beta, xc, yc = float(rng.uniform(3.0, 6.0)), float(rng.uniform(0, 10)), float(rng.uniform(0, 10))
    x = (torch.arange(nx, dtype=F64, device=dev) + 0.5) * (10.0 / nx) - xc
    y = (torch.arange(ny, dtype=F64, device=dev) + 0.5) * (10.0 / ny) - yc
    x = (x - 10.0 * torch.round(x / 10.0))[None, :]
    y = (y - 10.0 * torch.round(y / 10.0))[:, None]
    e = torch.exp(0.5 * (1.0 - x * x - y * y))
    u = 0.5 * math.sqrt(GAMMA) - beta / (2.0 * math.pi) * y * e
    v = beta / (2.0 * math.pi) * x * e
    T = 1.0 - (GAMMA - 1.0) * beta ** 2 / (8.0 * GAMMA * math.pi ** 2) * e * e
    r = T ** (1.0 / (GAMMA - 1.0))
    return [f[None].expand(nz, ny, nx) for f in (r, u, v, r * T)]


def _state(case, seed):
    """the conserved state of a flow case, [5][nz][ny][nx] float64 on the GPU"""
    dev, shape = _device(), _extent(case)
    rng = np.random.Generator(np.random.PCG64([1710, int(seed)]))
    if case["kind"] in ("block", "wcns") and case["viscous"]:
        r, u, v, p = _vortex(shape, rng, dev)
        w = _waves(shape, rng, 0.02, dev)
        return _conserved(r * (1.0 + _waves(shape, rng, 0.02, dev)), u, v, w, p * (1.0 + _waves(shape, rng, 0.02, dev)))
    if case["kind"] in ("block", "wcns"):  # Gaussian pulse in a Mach 0.5 stream on the unit box
        c = rng.random(3)
        d = []
        for n, x0 in zip(shape, c):
            x = (torch.arange(n, dtype=F64, device=dev) + 0.5) / n - float(x0)
            d.append((x - torch.round(x)) ** 2)
        g = 1e-2 * torch.exp(-(d[2][:, None, None] + d[1][None, :, None] + d[0][None, None, :]) / 0.01)
        z = torch.zeros_like(g)
        return _conserved(1.0 + g, z + 0.5, z, z, (1.0 + g) / GAMMA)
    mach = {"lattice": 0.8, "warped": 0.3, "channel": 0.6}[case["kind"]]
    amp = {"lattice": 1e-2, "warped": 0.05, "channel": 0.02}[case["kind"]]
    a = [_waves(shape, rng, amp, dev) for _ in range(5)]
    return _conserved(1.0 + a[0], mach + a[1], a[2], a[3], (1.0 + a[4]) / GAMMA)


def _spacing(case):
    nx, ny, nz = _extent(case)
    if case["kind"] == "lattice":
        return (1.0 / nx,) * 3
    if case["viscous"]:  # the vortex's 10 x 10 box, cells of the y size along z
        return (10.0 / nx, 10.0 / ny, 10.0 / ny)
    return (1.0 / nx, 1.0 / ny, 1.0 / nz)


def _viscosity(case):
    if not case.get("viscous"):
        return 0.0
    return 0.3 / 1e5 if case["kind"] == "warped" else 0.5 * math.sqrt(GAMMA) / 1e4


def _nodes(case, dev):
    """grid points [3][nz+1][ny+1][nx+1] of the curvilinear cases"""
    nx, ny, nz = _extent(case)
    x, y, z = (torch.arange(n + 1, dtype=F64, device=dev) / n for n in (nx, ny, nz))
    out = torch.empty((3, nz + 1, ny + 1, nx + 1), dtype=F64, device=dev)
    X, Y, Z = x[None, None, :], y[None, :, None], z[:, None, None]
    if case["kind"] == "warped":
        s = lambda a: torch.sin(2.0 * math.pi * a)
        out[0] = X + 0.05 * s(Y) * s(Z)
        out[1] = Y + 0.05 * s(Z) * s(X)
        out[2] = Z + 0.05 * s(X) * s(Y)
        return out
    # channel: x in [-1, 2], a sin^2 bump of height 0.1 on [0, 1], rows stretched away from the wall
    xs = -1.0 + 3.0 * X
    wall = torch.where((xs >= 0.0) & (xs <= 1.0), 0.1 * torch.sin(math.pi * xs) ** 2, torch.zeros_like(xs))
    eta = torch.expm1(3.0 * Y) / math.expm1(3.0)
    out[0] = xs.expand(nz + 1, ny + 1, nx + 1)
    out[1] = wall + (1.0 - wall) * eta
    out[2] = 0.5 * Z
    return out


CHANNEL_INF = (1.0, 0.6, 0.0, 0.0, 1.0 / GAMMA)


def _params(case):
    cfl = 0.9 if case["kind"] == "channel" else 0.5
    return gbcfd.params(GAMMA, _viscosity(case), PRANDTL, cfl, EPS, bool(case.get("viscous")), case.get("limiter", 0),
                        gbcfd.FP64 if case["precision"] == "fp64" else gbcfd.MIXED, case["kind"] == "channel")


def _accel_inputs(case, seed):
    """features bf16 [cells][16] (10 used), targets f32 [cells][8] (5 used), parameters f32"""
    dev = _device()
    rng = np.random.Generator(np.random.PCG64([40677, int(seed)]))
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(rng.integers(1 << 31)))
    cells = case["nx"] * case["ny"] * case["nz"] * case["batch"]
    x = torch.zeros((cells, 16), dtype=torch.float32, device=dev)
    x[:, :10] = torch.randn((cells, 10), generator=gen, device=dev)
    t = torch.zeros((cells, 8), dtype=torch.float32, device=dev)
    t[:, :5] = torch.randn((cells, 5), generator=gen, device=dev)
    p = []
    for ci, co in zip(CHANNELS[:-1], CHANNELS[1:]):
        p.append((rng.standard_normal(co * ci * 27) * math.sqrt(2.0 / (27 * ci))).astype(np.float32))
        p.append((0.1 * rng.standard_normal(co)).astype(np.float32))
    return x.to(torch.bfloat16), t, np.concatenate(p)


def prepare(case, seed):
    if case["kind"] in ("accel_forward", "accel_train"):
        x, t, p = _accel_inputs(case, seed)
        acc = gbcfd.Accel(case["nx"], case["ny"], case["nz"], case["batch"])
        acc.set_params(p)
        return {"kind": case["kind"], "acc": acc, "x": x, "t": t,
                "y": torch.empty((x.shape[0], 8), dtype=torch.float32, device=x.device)}
    q, prm = _state(case, seed), _params(case)
    st = {"kind": case["kind"], "steps": case["steps"]}
    if case["kind"] == "lattice":
        sx, sy, sz = _slab_sizes(case)
        ox, oy, oz = (np.concatenate([[0], np.cumsum(s)]).tolist() for s in (sx, sy, sz))
        at, st["q"] = {}, []
        for k in range(len(sz)):
            for j in range(len(sy)):
                for i in range(len(sx)):
                    b = gbcfd.Block(sx[i], sy[j], sz[k], prm)
                    b.set_metrics(spacing=_spacing(case))
                    at[i, j, k] = b
                    st["q"].append(q[:, oz[k]:oz[k + 1], oy[j]:oy[j + 1], ox[i]:ox[i + 1]].contiguous())
        for (i, j, k), b in at.items():
            b.connect("+x", at[(i + 1) % len(sx), j, k])
            b.connect("+y", at[i, (j + 1) % len(sy), k])
            b.connect("+z", at[i, j, (k + 1) % len(sz)])
        st["blocks"] = list(at.values())
        for b, part in zip(st["blocks"], st["q"]):
            b.set_state(part)
        st["group"] = gbcfd.Group(st["blocks"])
        st["group"].tune()
        st["out"] = [torch.empty_like(part) for part in st["q"]]
        return st
    nx, ny, nz = _extent(case)
    if case["kind"] == "wcns":
        b = gbcfd.WcnsBlock(nx, ny, nz, prm, _spacing(case))
    else:
        b = gbcfd.Block(nx, ny, nz, prm)
        if case["kind"] == "channel":
            for face, kind in (("-x", gbcfd.BC_FARFIELD), ("+x", gbcfd.BC_FARFIELD), ("-y", gbcfd.BC_SLIP_WALL),
                               ("+y", gbcfd.BC_SLIP_WALL)):
                b.set_boundary(face, kind, CHANNEL_INF)
            b.connect("+z", b)
        else:
            b.periodic()
        if case["kind"] == "block":
            b.set_metrics(spacing=_spacing(case))
        else:
            b.set_metrics(nodes=_nodes(case, q.device))
    st.update(block=b, q=q, out=torch.empty_like(q))
    b.set_state(q)
    return st


def run(state):
    kind = state["kind"]
    if kind == "accel_forward":
        return state["acc"].forward(state["x"], state["y"])
    if kind == "accel_train":
        loss = state["acc"].train_step(state["x"], state["t"], LR)
        grad, m, v = state["acc"].train_state()
        return {"loss": loss, "params": state["acc"].get_params(), "grad": grad, "m": m, "v": v}
    if kind == "lattice":
        for b, q in zip(state["blocks"], state["q"]):
            b.set_state(q)
        state["group"].step(state["steps"])
        return [b.get_state(o) for b, o in zip(state["blocks"], state["out"])]
    b = state["block"]
    b.set_state(state["q"])
    if kind == "wcns":
        b.step(state["steps"])
        return b.get_state(state["out"])
    gbcfd.step([b], state["steps"])
    if kind == "channel":
        norm = b.residual_norm()
        return {"state": b.get_state(state["out"]), "norm": norm}
    return b.get_state(state["out"])


def work(case):
    """bytes: the state in and out (and the nodes of a curvilinear grid; the accelerator's features,
    outputs and targets); flops: the schemes' floating-point operations per cell and stage (three
    faces of reconstruction, Roe and viscous flux, and the update), the network's multiply-adds"""
    if case["kind"] in ("accel_forward", "accel_train"):
        cells = case["nx"] * case["ny"] * case["nz"] * case["batch"]
        macs = 27 * sum(a * b for a, b in zip(CHANNELS[:-1], CHANNELS[1:]))
        if case["kind"] == "accel_forward":
            return {"bytes": cells * (20.0 + 20.0), "flops": 2.0 * macs * cells}
        back = macs - 27 * CHANNELS[0] * CHANNELS[1]  # no gradient for the inputs
        return {"bytes": cells * (20.0 + 20.0), "flops": 2.0 * (2 * macs + back) * cells}
    nx, ny, nz = _extent(case)
    cells = float(nx) * ny * nz
    per = {"block": 960.0, "lattice": 960.0, "warped": 1150.0, "channel": 1150.0, "wcns": 1400.0}[case["kind"]]
    if case.get("viscous"):
        per += {"wcns": 350.0, "warped": 400.0}.get(case["kind"], 110.0)
    grid = 24.0 if case["kind"] in ("warped", "channel") else 0.0
    return {"bytes": cells * (80.0 + grid), "flops": 3.0 * case["steps"] * per * cells}


# ---- the schemes in plain float64 --------------------------------------------------------------

def _prim(q):
    u = q[1:4] / q[0]
    p = (GAMMA - 1.0) * (q[4] - 0.5 * q[0] * (u * u).sum(0))
    return torch.cat([q[:1], u, p[None]])


def _cons(w):
    return _conserved(w[0], w[1], w[2], w[3], w[4])


def _cut(a, d, lo, n, core=2):
    """n entries of a padded array from `lo` along direction d (0 = x), interior ones along the others"""
    for e in range(3):
        ax = a.dim() - 1 - e
        a = a.narrow(ax, lo, n) if e == d else a.narrow(ax, core, a.shape[ax] - 2 * core)
    return a


def _wrap(a, d, n=2):
    ax = a.dim() - 1 - d
    if a.shape[ax] < n:
        idx = (torch.arange(-n, a.shape[ax] + n, device=a.device)) % a.shape[ax]
        return a.index_select(ax, idx)
    return torch.cat([a.narrow(ax, a.shape[ax] - n, n), a, a.narrow(ax, 0, n)], ax)


def _minmod(a, b):
    return torch.where(a * b > 0, torch.where(a.abs() < b.abs(), a, b), torch.zeros_like(a))


def _roe(l, r, S):
    """Roe flux with Harten's fix through area vectors S [3][...]; l, r primitives"""
    area = (S * S).sum(0).sqrt()
    n = S / area
    dot = lambda w: w[1] * n[0] + w[2] * n[1] + w[3] * n[2]
    ul, ur = dot(l), dot(r)
    h = lambda w: GAMMA / (GAMMA - 1.0) * w[4] / w[0] + 0.5 * (w[1:4] * w[1:4]).sum(0)
    hl, hr = h(l), h(r)
    flux = lambda w, un, hh: torch.stack([w[0] * un, w[0] * w[1] * un + w[4] * n[0], w[0] * w[2] * un + w[4] * n[1],
                                          w[0] * w[3] * un + w[4] * n[2], w[0] * hh * un])
    F = flux(l, ul, hl) + flux(r, ur, hr)
    sl, sr = l[0].sqrt(), r[0].sqrt()
    rho = sl * sr
    mean = lambda a, b: (sl * a + sr * b) / (sl + sr)
    v, ht = mean(l[1:4], r[1:4]), mean(hl, hr)
    q2 = (v * v).sum(0)
    c2 = (GAMMA - 1.0) * (ht - 0.5 * q2)
    c = c2.sqrt()
    un = (v * n).sum(0)
    dr, dp, du, dun = r[0] - l[0], r[4] - l[4], r[1:4] - l[1:4], ur - ul
    a1, a5, a2 = (dp - rho * c * dun) / (2.0 * c2), (dp + rho * c * dun) / (2.0 * c2), dr - dp / c2
    sh = rho * (du - dun * n)
    delta = EPS * (un.abs() + c)
    fix = lambda x: torch.where(x.abs() < delta, (x * x + delta * delta) / (2.0 * delta), x.abs())
    w1, w2, w5, l2 = fix(un - c) * a1, fix(un) * a2, fix(un + c) * a5, fix(un)
    F[0] -= w1 + w2 + w5
    F[1:4] -= w1 * (v - c * n) + w2 * v + l2 * sh + w5 * (v + c * n)
    F[4] -= w1 * (ht - c * un) + w2 * 0.5 * q2 + l2 * (v * sh).sum(0) + w5 * (ht + c * un)
    return 0.5 * area * F


def _grid(case, dev):
    """padded metrics: lower-face area vectors [3][3][..] and volumes [..] (expanded views where uniform)"""
    nx, ny, nz = _extent(case)
    shape = (nz + 4, ny + 4, nx + 4)
    if case["kind"] not in ("warped", "channel"):
        h = _spacing(case)
        S = torch.zeros((3, 3, 1, 1, 1), dtype=F64, device=dev)
        for d in range(3):
            S[d, d] = h[(d + 1) % 3] * h[(d + 2) % 3]
        V = torch.full((1, 1, 1), h[0] * h[1] * h[2], dtype=F64, device=dev)
        return S.expand((3, 3) + shape), V.expand(shape)
    X = _nodes(case, dev)
    if case["kind"] == "channel":  # nodes beyond x and y boundaries: reflected through the boundary node
        for d in (0, 1):
            ax, n = 3 - d, X.shape[3 - d] - 1
            at = lambda i: X.narrow(ax, i, 1)
            X = torch.cat([2 * at(0) - at(2), 2 * at(0) - at(1), X, 2 * at(n) - at(n - 1), 2 * at(n) - at(n - 2)], ax)
    K, J, I = (s - 1 for s in X.shape[1:])
    c = lambda dk, dj, di: X[:, dk:dk + K, dj:dj + J, di:di + I]
    quad = lambda a, b, e, f: 0.5 * torch.linalg.cross(e - a, f - b, dim=0)
    faces = {  # lower and upper corners of the faces towards +x, +y, +z
        0: [(c(0, 0, i), c(0, 1, i), c(1, 1, i), c(1, 0, i)) for i in (0, 1)],
        1: [(c(0, j, 0), c(1, j, 0), c(1, j, 1), c(0, j, 1)) for j in (0, 1)],
        2: [(c(k, 0, 0), c(k, 0, 1), c(k, 1, 1), c(k, 1, 0)) for k in (0, 1)]}
    V, S = 0.0, []
    for d in range(3):
        for side, f in enumerate(faces[d]):
            s = quad(*f)
            if side == 0:
                S.append(s)
            V = V + (2 * side - 1) * ((sum(f) / 4.0 - c(0, 0, 0)) * s).sum(0)
    S, V = torch.stack(S), V / 3.0
    for d in ((2,) if case["kind"] == "channel" else (0, 1, 2)):
        S, V = _wrap(S, d), _wrap(V, d)
    return S, V


def _padded(case, q, S):
    """primitives of the interior state q with two halo cells on every side"""
    w = _prim(q)
    if case["kind"] != "channel":
        for d in range(3):
            w = _wrap(w, d)
        return w
    w = _wrap(w, 2)
    inf = torch.tensor(CHANNEL_INF, dtype=F64, device=q.device)[:, None, None]
    nx, ny = q.shape[3], q.shape[2]

    def far(wi, n):  # characteristic far field, outward normal n
        ci, ce = (GAMMA * wi[4] / wi[0]).sqrt(), math.sqrt(GAMMA * CHANNEL_INF[4] / CHANNEL_INF[0])
        un, ue = (wi[1:4] * n).sum(0), CHANNEL_INF[1] * n[0] + CHANNEL_INF[2] * n[1] + CHANNEL_INF[3] * n[2]
        rp, rm = un + 2.0 * ci / (GAMMA - 1.0), ue - 2.0 * ce / (GAMMA - 1.0)
        ub, cb = 0.5 * (rp + rm), 0.25 * (GAMMA - 1.0) * (rp - rm)
        src = torch.where(ub < 0.0, inf, wi)
        us = (src[1:4] * n).sum(0)
        r = (cb * cb / (GAMMA * src[4] / src[0] ** GAMMA)) ** (1.0 / (GAMMA - 1.0))
        out = torch.cat([r[None], src[1:4] + (ub - us) * n, (r * cb * cb / GAMMA)[None]])
        out = torch.where((un >= ci)[None], wi, out)
        return torch.where((ue <= -ce)[None], inf.expand_as(out), out)

    unit = lambda s: s / (s * s).sum(0).sqrt()
    lo = far(w[..., 0], -unit(S[0, :, :, 2:-2, 2]))
    hi = far(w[..., nx - 1], unit(S[0, :, :, 2:-2, nx + 2]))
    w = torch.cat([lo[..., None], lo[..., None], w, hi[..., None], hi[..., None]], 3)

    def mirror(wi, n):
        un = (wi[1:4] * n).sum(0)
        return torch.cat([wi[:1], wi[1:4] - 2.0 * un * n, wi[4:]])[:, :, None]

    lo, hi = unit(S[1, :, :, 2, :]), unit(S[1, :, :, ny + 2, :])
    m = lambda j, n: mirror(w[:, :, j], n)
    return torch.cat([m(1, lo), m(0, lo), w, m(ny - 1, hi), m(ny - 2, hi)], 2)


def _viscous(w, S, V, d, mu):
    n = w.shape[3 - d] - 4
    phi = torch.cat([w[1:4], (w[4] / w[0])[None]])

    def at(a, side, d2=None, off=0):  # the face's left (0) or right (1) cell, shifted by off along d2
        for e in range(3):
            ax = a.dim() - 1 - e
            a = a.narrow(ax, 1 + side, n + 1) if e == d else a.narrow(ax, 2 + (off if e == d2 else 0), a.shape[ax] - 4)
        return a

    L, R = at(phi, 0), at(phi, 1)
    g = (R - L)[:, None] * at(S[d], 1)[None]
    for t in ((d + 1) % 3, (d + 2) % 3):
        dt = 0.25 * sum(at(phi, s, t, 1) - at(phi, s, t, -1) for s in (0, 1))
        Sb = 0.25 * sum(at(S[t], s) + at(S[t], s, t, 1) for s in (0, 1))
        g += dt[:, None] * Sb[None]
    g /= 0.5 * (at(V, 0) + at(V, 1))
    div = g[0, 0] + g[1, 1] + g[2, 2]
    Sf = at(S[d], 1)
    tS = torch.stack([sum(mu * (g[r, s] + g[s, r]) * Sf[s] for s in range(3)) - 2.0 / 3.0 * mu * div * Sf[r] for r in range(3)])
    kappa = mu * GAMMA / ((GAMMA - 1.0) * PRANDTL)
    e = (0.5 * (L[:3] + R[:3]) * tS).sum(0) + kappa * (g[3] * Sf).sum(0)
    return torch.cat([torch.zeros_like(e)[None], tS, e[None]])


def _residual(case, q, S, V):
    w = _padded(case, q, S)
    total = torch.zeros_like(q)
    for d in range(3):
        n = q.shape[3 - d]
        s = [_cut(w, d, o, n + 1) for o in range(4)]
        if case.get("limiter", 0):
            l, r = s[1] + 0.25 * (s[2] - s[0]), s[2] - 0.25 * (s[3] - s[1])
        else:
            l, r = s[1] + 0.5 * _minmod(s[1] - s[0], s[2] - s[1]), s[2] - 0.5 * _minmod(s[2] - s[1], s[3] - s[2])
        F = _roe(l, r, _cut(S[d], d, 2, n + 1))
        if case.get("viscous"):
            F -= _viscous(w, S, V, d, _viscosity(case))
        total += F.narrow(3 - d, 1, n) - F.narrow(3 - d, 0, n)
    return total / _cut(V, 0, 2, V.shape[2] - 4)


def _rate(case, q, S, V):
    """sum over directions of the spectral radii over the volume, per cell"""
    w = _prim(q)
    a = (GAMMA * w[4] / w[0]).sqrt()
    vol = V[2:-2, 2:-2, 2:-2]
    rate = 0.0
    for d in range(3):
        n = q.shape[3 - d]
        Sb = 0.5 * (_cut(S[d], d, 2, n) + _cut(S[d], d, 3, n))
        s2 = (Sb * Sb).sum(0)
        rate = rate + (w[1:4] * Sb).sum(0).abs() + a * s2.sqrt()
        if case.get("viscous"):
            rate = rate + 4.0 * max(4.0 / 3.0, GAMMA / PRANDTL) * _viscosity(case) / w[0] * s2 / vol
    return rate / vol


def _wcns_residual(case, q, h):
    w = _prim(q)
    roll = lambda a, d, s: torch.roll(a, -s, a.dim() - 1 - d)  # the value s cells further along d
    mu = _viscosity(case)
    total = torch.zeros_like(q)
    for d in range(3):
        def edge(u):
            g = [0.5 * (u[0] - 4.0 * u[1] + 3.0 * u[2]), 0.5 * (u[3] - u[1]), 0.5 * (-3.0 * u[2] + 4.0 * u[3] - u[4])]
            s = [u[0] - 2.0 * u[1] + u[2], u[1] - 2.0 * u[2] + u[3], u[2] - 2.0 * u[3] + u[4]]
            C = (1.0 / 16.0, 10.0 / 16.0, 5.0 / 16.0)
            if case.get("limiter", 0):
                a = [torch.full_like(u[0], c) for c in C]
            else:
                a = [c / (WCNS_EPS + gk * gk + sk * sk) ** 2 for c, gk, sk in zip(C, g, s)]
            return u[2] + sum(ak * (0.5 * gk + 0.125 * sk) for ak, gk, sk in zip(a, g, s)) / sum(a)

        l, r = edge([roll(w, d, o) for o in (-2, -1, 0, 1, 2)]), edge([roll(w, d, o) for o in (3, 2, 1, 0, -1)])
        n = torch.zeros((3, 1, 1, 1), dtype=F64, device=q.device)
        n[d] = 1.0
        F = _roe(l, r, n)
        for c, o in ((75.0 / 64.0, 0), (-25.0 / 384.0, 1), (3.0 / 640.0, 2)):
            total += (roll(F, d, o) - roll(F, d, -1 - o)) * (c / h[d])
    if mu:
        d4 = lambda a, d: (roll(a, d, -2) - 8.0 * roll(a, d, -1) + 8.0 * roll(a, d, 1) - roll(a, d, 2)) / (12.0 * h[d])
        phi = torch.cat([w[1:4], (w[4] / w[0])[None]])
        g = [d4(phi, d) for d in range(3)]  # g[d][q]
        div = g[0][0] + g[1][1] + g[2][2]
        kappa = mu * GAMMA / ((GAMMA - 1.0) * PRANDTL)
        for d in range(3):
            tau = [mu * (g[d][a] + g[a][d]) - (2.0 / 3.0 * mu * div if a == d else 0.0) for a in range(3)]
            e = sum(w[1 + a] * tau[a] for a in range(3)) + kappa * g[d][3]
            total[1:] -= d4(torch.stack(tau + [e]), d)
    return total


def _march(case, q):
    if case["kind"] == "wcns":
        h = _spacing(case)
        res = lambda x: _wcns_residual(case, x, h)
        S, V = _grid(case, q.device)
    else:
        S, V = _grid(case, q.device)
        res = lambda x: _residual(case, x, S, V)
    norm = None
    for _ in range(case["steps"]):
        rate = _rate(case, q, S, V)
        dt = 0.9 / rate if case["kind"] == "channel" else 0.5 / rate.max()
        R = res(q)
        norm = (R * R).mean((1, 2, 3)).sqrt()
        q1 = q - dt * R
        q2 = 0.75 * q + 0.25 * (q1 - dt * res(q1))
        q = q / 3.0 + 2.0 / 3.0 * (q2 - dt * res(q2))
    return q, norm


def _network(case, x, params):
    """x [batch][10][z][y][x], params a list of (weight, bias); zero padding in x and y, periodic in z"""
    for i, (W, b) in enumerate(params):
        x = torch.nn.functional.pad(torch.cat([x[:, :, -1:], x, x[:, :, :1]], 2), (1, 1, 1, 1))
        k, j, l = (s - 2 for s in x.shape[2:])
        y = b[None, :, None, None, None]
        for t in range(27):
            dz, dy, dx = t // 9, t // 3 % 3, t % 3
            y = y + torch.einsum("oc,bczyx->bozyx", W[:, :, t], x[:, :, dz:dz + k, dy:dy + j, dx:dx + l])
        x = y * torch.sigmoid(y) if i < 2 else y
    return x


def _exact_accel(case, seed):
    x, t, p = _accel_inputs(case, seed)
    p = torch.from_numpy(p).to(x.device).to(F64).requires_grad_(case["kind"] == "accel_train")
    params, o = [], 0
    for ci, co in zip(CHANNELS[:-1], CHANNELS[1:]):
        params.append((p[o:o + co * ci * 27].view(co, ci, 27), p[o + co * ci * 27:o + co * ci * 27 + co]))
        o += co * ci * 27 + co
    vol = (case["batch"], case["nz"], case["ny"], case["nx"])
    y = _network(case, x[:, :10].to(F64).view(vol + (10,)).permute(0, 4, 1, 2, 3), params)
    y = y.permute(0, 2, 3, 4, 1).reshape(-1, 5)
    if case["kind"] == "accel_forward":
        return torch.cat([y, torch.zeros((y.shape[0], 3), dtype=F64, device=y.device)], 1)
    loss = ((y - t[:, :5].to(F64)) ** 2).mean()
    g, = torch.autograd.grad(loss, p)
    m, v = 0.1 * g, 0.001 * g * g
    new = p.detach() - LR * (m / 0.1) / ((v / 0.001).sqrt() + 1e-8)
    as_np = lambda a: a.detach().cpu().numpy()
    return {"loss": float(loss), "params": as_np(new), "grad": as_np(g), "m": as_np(m), "v": as_np(v)}


def exact(case, seed):
    if case["kind"] in ("accel_forward", "accel_train"):
        return _exact_accel(case, seed)
    q, norm = _march(case, _state(case, seed))
    if case["kind"] == "channel":
        return {"state": q, "norm": norm.cpu().numpy()}
    if case["kind"] != "lattice":
        return q
    sx, sy, sz = (np.concatenate([[0], np.cumsum(s)]).tolist() for s in _slab_sizes(case))
    return [q[:, sz[k]:sz[k + 1], sy[j]:sy[j + 1], sx[i]:sx[i + 1]].contiguous()
            for k in range(len(sz) - 1) for j in range(len(sy) - 1) for i in range(len(sx) - 1)]
