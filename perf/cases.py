"""Workloads of the MHD library as its users run them, for timing and for
checking results against plain FP64.

A case is a dict of plain values; its "kind" says which public calls a pass
makes:

  box       mhd.Box: state in, a device-resident CFL run of `steps` full
            steps, state out (restart, advance, read back)
  ensemble  mhd.Ensemble: the same for `count` uneven boxes advanced together
  box64     mhd.Box64: the FP64 path
  diag      Box.diagnostics of a state that is already in the box
  restrict  mhd.restrict of a fine state by r along every axis
  coarse    one learned coarse step: predict, step, corrected state
  train     forward, loss and gradients of the correction network

`exact` repeats a pass in FP64 with plain torch operations from the scheme's
definition (relaxing-TVD fluid sweeps, constrained-transport magnetic sweeps,
[F_d M_d] for d = x, y, z and [M_d F_d] for d = z, y, x).
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_1004_1680_gb300 import initial_conditions as ic
from paper_1004_1680_gb300 import learned, mhd

GAMMA = 5.0 / 3.0
CFL = 0.7
GHOST = 4  # ghost cells at each end of a non-periodic axis
MODES = {"p": "periodic", "o": "outflow", "r": "reflecting"}


def _box(nx, ny, nz, steps, bc="ppp", floor=0.0, ic="turbulence", mach=1.0, beta=1.0):
    return {"kind": "box", "nx": nx, "ny": ny, "nz": nz, "steps": steps, "bc": bc, "floor": floor, "ic": ic,
            "mach": mach, "beta": beta}


def listed():
    cases = {
        # the smallest box the paper times and the tests use throughout: launches and latency
        "box 32^3": _box(32, 32, 32, 20),
        # a one-dimensional shock tube between open ends (the pins' workload): few pencils, ghost layers
        "tube 512x8x8": _box(512, 8, 8, 40, bc="opp", ic="tube"),
        # the largest box the paper times
        "box 128^3": _box(128, 128, 128, 10),
        # an odd box with open walls and the pressure floor, as a run of a region would be set up
        "walls 236x150x98": _box(236, 150, 98, 6, bc="poo", floor=1e-3, mach=0.5, beta=4.0),
        # the fine box behind every training pair and comparison run of the learned correction
        "box 256^3": _box(256, 256, 256, 4, floor=1e-3),
        # the benchmark's box
        "box 512^3": _box(512, 512, 512, 3),
        # the benchmark's ensemble recipe (uneven boxes, Mach and beta by box) with fewer boxes
        "ensemble 32": {"kind": "ensemble", "count": 32, "dims_seed": 2024, "steps": 16, "floor": 1e-3},
        # the FP64 path on a box a convergence or precision study would take
        "box64 64^3": {"kind": "box64", "nx": 64, "ny": 64, "nz": 64, "steps": 3},
        # conservation sums, div b and min p of the fine box (monitoring between runs)
        "diagnostics 256^3": {"kind": "diag", "nx": 256, "ny": 256, "nz": 256},
        # fine state to coarse state, once per training pair and comparison sample
        "restrict 256^3": {"kind": "restrict", "nx": 256, "ny": 256, "nz": 256, "r": 4},
        # one step of the learned 64^3 run: CFL timestep, prediction, step, clipped correction
        "learned step 64^3": {"kind": "coarse", "nx": 64, "ny": 64, "nz": 64},
        # one training pair of the correction network up to its gradients
        "gradients 64^3": {"kind": "train", "nx": 64, "ny": 64, "nz": 64},
    }
    return [dict(c, name=name) for name, c in cases.items()]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["box"] * 5 + ["ensemble", "box64", "diag", "restrict", "coarse", "train"])
    if kind in ("coarse", "train"):
        return {"kind": kind, "nx": 8 * rng.randint(2, 16), "ny": 16 * rng.randint(1, 8), "nz": rng.randint(12, 100)}
    if kind == "restrict":
        r = rng.choice([2, 3, 4])
        return {"kind": kind, "nx": r * rng.randint(6, 90), "ny": r * rng.randint(6, 90), "nz": r * rng.randint(6, 90),
                "r": r}
    if kind == "ensemble":
        return {"kind": kind, "count": rng.randint(3, 48), "dims_seed": rng.randrange(1 << 20),
                "steps": rng.randint(2, 12), "floor": 1e-3}
    cells = _log_uniform(rng, 16 ** 3, 140 ** 3 if kind == "box64" else 420 ** 3)
    side = cells ** (1.0 / 3.0)
    nx = side * _log_uniform(rng, 0.5, 2.0)
    ny = side * _log_uniform(rng, 0.6, 1.7)
    # half of the boxes have the round x extents that users pick, the others any multiple of 4
    whole = [n for n in (16, 32, 64, 128, 256, 384, 512) if 0.6 * nx <= n <= 1.7 * nx]
    nx = rng.choice(whole) if whole and rng.random() < 0.5 else 4 * max(3, round(nx / 4))
    ny = max(12, round(ny) if rng.random() < 0.5 else 8 * round(ny / 8))
    nz = max(12, round(cells / (nx * ny)))
    if kind == "diag":
        return {"kind": kind, "nx": nx, "ny": ny, "nz": nz}
    if kind == "box64":
        return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "steps": rng.randint(1, 3)}
    steps = max(1, min(20, int(2.0e8 / (nx * ny * nz))))
    bc = rng.choice(["ppp", "ppp", "ppp", "ppo", "opp", "ooo"])
    return _box(nx, ny, nz, steps, bc=bc, floor=1e-3 if bc != "ppp" else rng.choice([0.0, 1e-3]),
                mach=0.5 if bc != "ppp" else round(rng.uniform(0.3, 1.0), 3), beta=4.0 if bc != "ppp" else 1.0)


# --------------------------------------------------------------------------
# inputs

def _turbulence(n, seed, mach, beta, dtype=torch.float32):
    # wavelengths of 8 cells and more, at most the recipe's k = 8
    return ic.turbulence(n, seed=seed, mach=mach, beta=beta, device="cuda", dtype=dtype, kmin=1.0,
                         kmax=max(1.5, min(8.0, min(n) / 8.0)))


def _tube(n, seed):
    """A Brio-Wu-like tube along x, its left state varied by the seed."""
    nx, ny, nz = n
    rng = np.random.default_rng(seed)
    left = torch.arange(nx, device="cuda") < nx // 2
    f = lambda a, b: torch.where(left, float(a), float(b)).double().expand(nz, ny, nx).contiguous()  # noqa: E731
    s = 1.0 + 0.1 * rng.uniform(-1.0, 1.0, size=2)
    zero = f(0.0, 0.0)
    return ic.assemble(f(s[0], 0.125), [zero, f(0.1 * (s[1] - 1.0), 0.0), zero], f(s[1], 0.1),
                       [f(0.75, 0.75), f(1.0, -1.0), zero], dtype=torch.float32)


def _state(case, seed, dtype=torch.float32):
    n = (case["nx"], case["ny"], case["nz"])
    if case.get("ic") == "tube":
        return _tube(n, seed)
    return _turbulence(n, seed, case.get("mach", 1.0), case.get("beta", 1.0), dtype)


def _ensemble_states(case, seed):
    specs = ic.ensemble_specs(case["count"], seed=case["dims_seed"])
    return [(s["dims"], _turbulence(s["dims"], 1000 * seed + s["seed"], s["mach"], s["beta"])) for s in specs]


def _network(seed):
    """He-initialised weights as CorrectionNet makes them, small biases (a
    trained network has some), the last layer scaled down."""
    g = torch.Generator().manual_seed(seed + 17)
    W, b = [], []
    for li, (ci, co) in enumerate(learned.LAYERS):
        std = math.sqrt(2.0 / (27 * ci)) * (0.1 if li == 3 else 1.0)
        W.append(torch.randn(co, ci, 3, 3, 3, generator=g) * std)
        b.append(torch.randn(co, generator=g) * 0.02)
    return [w.cuda() for w in W], [x.cuda() for x in b]


def _norm(state):
    """Input normalisation by the state's own fields; corrections of a
    thousandth of their spread, as one coarse step needs."""
    x = state.double()
    sd = x.std(dim=(1, 2, 3)).clamp_min(1e-2)
    ts = (1e-3 * sd).tolist()
    return learned.Norm(mu=x.mean(dim=(1, 2, 3)).tolist(), inv_sigma=(1.0 / sd).tolist(),
                        out_scale=ts[:5] + [float(np.mean(ts[5:8])) / state.shape[-1]],
                        loss_weight=[1.0 / (8.0 * t * t * state[0].numel()) for t in ts])


def _target(state, norm, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + 5)
    t = torch.randn(state.shape, generator=g, device="cuda", dtype=torch.float32)
    w = torch.tensor([1.0 / math.sqrt(8.0 * x * state[0].numel()) for x in norm.loss_weight], device="cuda")
    return t * w.view(8, 1, 1, 1)


# --------------------------------------------------------------------------
# a pass

def _make_net(W, b):
    net = learned.CorrectionNet(seed=0)
    for mine, given in zip(net.W + net.b, W + b):
        mine.copy_(given)
    net.repack()
    return net


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": dict(case)}
    if kind == "ensemble":
        states = _ensemble_states(case, seed)
        ens = mhd.Ensemble([d for d, _ in states])
        ens.set_pressure_floor(case["floor"])
        st["states"] = [s for _, s in states]
        for i, s in enumerate(st["states"]):
            ens.set_state(i, s)
        ens.autotune(CFL)
        st["ens"] = ens
        return st
    n = (case["nx"], case["ny"], case["nz"])
    st["x"] = _state(case, seed, torch.float64 if kind == "box64" else torch.float32)
    if kind == "box64":
        st["box"] = mhd.Box64(*n)
    elif kind in ("box", "diag", "coarse"):
        st["box"] = box = mhd.Box(*n)
        st["out"] = torch.empty_like(st["x"])
        if kind == "box":
            for axis, mode in enumerate(case["bc"]):
                if mode != "p":
                    box.set_boundary(axis, MODES[mode])
            box.set_pressure_floor(case["floor"])
        if kind == "diag":
            box.set_state(st["x"])
    if kind in ("coarse", "train"):
        norm = _norm(st["x"])
        st["corr"] = learned.Corrector(_make_net(*_network(seed)), norm, n)
    if kind == "train":
        st["target"] = _target(st["x"], norm, seed)
        st["g"] = torch.empty_like(st["corr"].d)
        st["loss"] = torch.empty(1, dtype=torch.float64, device="cuda")
        st["gy"] = torch.empty((n[0] * n[1] * n[2], 8), dtype=torch.bfloat16, device="cuda")
        st["sums"] = torch.empty(5, dtype=torch.float64, device="cuda")
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "box":
        box = st["box"]
        box.set_state(st["x"])
        box.run(case["steps"], CFL)
        if case["bc"] != "ppp":
            box.fill_ghosts()
        return box.get_state(out=st["out"])
    if kind == "ensemble":
        ens = st["ens"]
        for i, s in enumerate(st["states"]):
            ens.set_state(i, s)
        ens.run(case["steps"], CFL)
        return [ens.get_state(i) for i in range(len(st["states"]))]
    if kind == "box64":
        box = st["box"]
        box.set_state(st["x"])
        box.run(case["steps"], CFL)
        return box.get_state()
    if kind == "diag":
        return st["box"].diagnostics()
    if kind == "restrict":
        return mhd.restrict(st["x"], case["r"])
    corr, n = st["corr"], (case["nx"], case["ny"], case["nz"])
    if kind == "coarse":
        box = st["box"]
        box.set_state(st["x"])
        dt = box.cfl_dt(CFL)
        d = corr.predict(st["x"])
        box.step(dt)
        s = box.get_state(out=st["out"])
        corr.apply(s, d)
        box.set_state(s)
        return {"state": s, "correction": d}
    norm, net = corr.norm, corr.net
    mhd.cnn_normalize(st["x"], norm.mu, norm.inv_sigma, out=corr.x)
    y, acts = net.forward(corr.x, n)
    d = mhd.cnn_project(y, n, norm.out_scale, out=corr.d, sums=corr.sums)
    mhd.cnn_loss(d, st["target"], norm.loss_weight, g=st["g"], loss=st["loss"])
    mhd.cnn_project_backward(st["g"], norm.out_scale, out=st["gy"], sums=st["sums"])
    net.backward(st["gy"], acts, n)
    # the last bias's gradient is zero but for rounding (the projection removes the means it would move)
    return {"correction": d, "loss": st["loss"], "grads": net.grads[:-1]}


# --------------------------------------------------------------------------
# what a pass cannot do without

OPS_PER_CELL_STEP = 2366  # the paper's operation count of a full step (CFL, 6 fluid and 6 magnetic updates)
MACS_PER_CELL = sum(27 * ci * co for ci, co in learned.LAYERS)


def work(case):
    kind = case["kind"]
    if kind == "ensemble":
        cells = sum(math.prod(s["dims"]) for s in ic.ensemble_specs(case["count"], seed=case["dims_seed"]))
    else:
        cells = case["nx"] * case["ny"] * case["nz"]
    if kind in ("box", "ensemble", "box64"):
        # every step depends on a maximum over the whole state of the step before: 8 fields in, 8 fields out
        per = 128 if kind == "box64" else 64
        return {"bytes": per * cells * case["steps"], "flops": OPS_PER_CELL_STEP * cells * case["steps"]}
    if kind == "diag":
        return {"bytes": 32 * cells, "flops": 40 * cells}
    if kind == "restrict":
        return {"bytes": 32 * (cells + cells // case["r"] ** 3), "flops": 8 * cells}
    if kind == "coarse":  # state in, corrected state and correction out
        return {"bytes": 96 * cells, "flops": (2 * MACS_PER_CELL + OPS_PER_CELL_STEP) * cells}
    # state and target in, correction out; forward, input gradients (not of the first layer), weight gradients
    return {"bytes": 96 * cells, "flops": 2 * (3 * MACS_PER_CELL - 27 * 8 * 32) * cells}


# --------------------------------------------------------------------------
# the same in FP64 with plain torch: fields (8, nz, ny, nx), axis d is array dimension -1 - d

def _next(a, d):
    return torch.roll(a, -1, -1 - d)


def _prev(a, d):
    return torch.roll(a, 1, -1 - d)


def _half_limiter(a, b):
    ab = a * b
    return torch.where(ab > 0, ab / torch.where(ab > 0, a + b, 1.0), 0.0)


def _centred(U):
    return [0.5 * (U[5 + d] + _next(U[5 + d], d)) for d in range(3)]


def _pressure(u, b):
    b2 = b[0] ** 2 + b[1] ** 2 + b[2] ** 2
    return (GAMMA - 1) * (u[4] - 0.5 * (u[1] ** 2 + u[2] ** 2 + u[3] ** 2) / u[0] - 0.5 * b2), b2


def _movers(u, b, d):
    p, b2 = _pressure(u, b)
    v = u[1 + d] / u[0]
    c = v.abs() + torch.sqrt((GAMMA * p + b2) / u[0])
    flux = u * v
    flux[0] = u[1 + d]
    flux[1 + d] += p + 0.5 * b2
    flux[4] += (p + 0.5 * b2) * v - b[d] * (b[0] * u[1] + b[1] * u[2] + b[2] * u[3]) / u[0]
    for a in range(3):
        flux[1 + a] -= b[d] * b[a]
    right = 0.5 * (c * u + flux)
    return right, right - flux


def _fluid(U, d, tau, floor):
    c = tau * U.shape[-1 - d]
    b = _centred(U)
    u = U[:5]
    R, L = _movers(u, b, d)
    f = R - _next(L, d)
    R, L = _movers(u - 0.5 * c * (f - _prev(f, d)), b, d)
    del f
    s = R - _prev(R, d)
    R += _half_limiter(s, _next(s, d))
    s = L - _prev(L, d)
    L -= _half_limiter(s, _next(s, d))
    del s
    f = R - _next(L, d)
    del R, L
    u -= c * (f - _prev(f, d))
    if floor > 0:
        p, _ = _pressure(u, b)
        u[4] += (floor - p).clamp_min(0.0) / (GAMMA - 1)


def _magnetic(U, d, tau):
    c = tau * U.shape[-1 - d]
    v = U[1 + d] / U[0]
    for t in ((d + 1) % 3, (d + 2) % 3):
        q = U[5 + t]
        face = 0.5 * (v + _prev(v, t))
        w = 0.5 * (face + _next(face, d))
        g = w * torch.where(w >= 0, q, _next(q, d))
        h = q - 0.5 * c * (g - _prev(g, d))
        s = h - _prev(h, d)
        s1 = _next(s, d)
        f = w * torch.where(w >= 0, h + _half_limiter(s, s1), _next(h, d) - _half_limiter(s1, _next(s1, d)))
        q -= c * (f - _prev(f, d))
        U[5 + d] += _prev(tau * U.shape[-1 - t] * (_next(f, t) - f), d)


def _fill_ghosts(U, bc):
    for a, mode in enumerate(bc):
        if mode == "p":
            continue
        n = U.shape[-1 - a]
        X = U.transpose(-1, -1 - a)  # a view with axis a last
        for g in range(GHOST):
            lo, hi = (GHOST, n - GHOST - 1) if mode == "o" else (2 * GHOST - 1 - g, n - 2 * GHOST + g)
            for q in range(8):
                if q == 5 + a:
                    continue
                sign = -1.0 if mode == "r" and q == 1 + a else 1.0
                X[q, ..., g] = sign * X[q, ..., lo]
                X[q, ..., n - 1 - g] = sign * X[q, ..., hi]
        for g in range(GHOST):
            k = n - 1 - g
            X[5 + a, ..., g] = X[5 + a, ..., GHOST] if mode == "o" else -X[5 + a, ..., 2 * GHOST - g]
            if k > n - GHOST:
                X[5 + a, ..., k] = X[5 + a, ..., n - GHOST] if mode == "o" else -X[5 + a, ..., 2 * (n - GHOST) - k]


def _rate(U, bc):
    b = _centred(U)
    p, b2 = _pressure(U, b)
    cf = torch.sqrt((GAMMA * p + b2) / U[0])
    r = None
    for d in range(3):
        x = ((U[1 + d] / U[0]).abs() + cf) * U.shape[-1 - d]
        r = x if r is None else torch.maximum(r, x)
    for a, mode in enumerate(bc):
        if mode != "p":
            r = r.narrow(-1 - a, GHOST, r.shape[-1 - a] - 2 * GHOST)
    return r.max()


def _step(U, tau, bc="ppp", floor=0.0):
    for d in (0, 1, 2):
        _fill_ghosts(U, bc)
        _fluid(U, d, tau, floor)
        _fill_ghosts(U, bc)
        _magnetic(U, d, tau)
    for d in (2, 1, 0):
        _fill_ghosts(U, bc)
        _magnetic(U, d, tau)
        _fill_ghosts(U, bc)
        _fluid(U, d, tau, floor)


def _advance(U, steps, bc="ppp", floor=0.0):
    for _ in range(steps):
        _fill_ghosts(U, bc)
        _step(U, CFL / _rate(U, bc), bc, floor)
    _fill_ghosts(U, bc)
    return U


class _Bf16(torch.autograd.Function):
    """Rounding to the network's operand type, of a value and of its gradient."""

    @staticmethod
    def forward(ctx, x):
        return x.to(torch.bfloat16).double()

    @staticmethod
    def backward(ctx, g):
        return g.to(torch.bfloat16).double()


def _conv(x, w, b):
    """3x3x3 periodic convolution as 27 matrix products: x (cin, nz, ny, nx)."""
    nz, ny, nx = x.shape[1:]
    p = F.pad(x.unsqueeze(0), (1,) * 6, mode="circular")[0]
    y = b.view(-1, 1)
    for k in range(3):
        for j in range(3):
            for i in range(3):
                y = y + w[:, :, k, j, i] @ p[:, k:k + nz, j:j + ny, i:i + nx].reshape(x.shape[0], -1)
    return y.view(-1, nz, ny, nx)


def _correction(x, norm, W, b, scale):
    """Network and projection; every operand of a convolution rounded to BF16."""
    mu, isig = (torch.tensor(v, dtype=torch.float32, device="cuda").view(8, 1, 1, 1) for v in (norm.mu, norm.inv_sigma))
    h = ((x - mu) * isig).to(torch.bfloat16).double()
    for li in range(4):
        h = _conv(h, W[li].detach().to(torch.bfloat16).double() - W[li].detach() + W[li], b[li])
        h = _Bf16.apply(torch.relu(h)) if li < 3 else _grad_bf16(h)
    nz, ny, nx = x.shape[1:]
    s = [float(np.float32(v)) for v in scale]
    cells = [s[q] * h[q] - (s[q] * h[q]).mean() for q in range(5)]
    ax, ay, az = (s[5] * h[5 + a] for a in range(3))
    curl = [(_next(az, 1) - az) * ny - (_next(ay, 2) - ay) * nz, (_next(ax, 2) - ax) * nz - (_next(az, 0) - az) * nx,
            (_next(ay, 0) - ay) * nx - (_next(ax, 1) - ax) * ny]
    return torch.stack(cells + curl)


class _GradBf16(torch.autograd.Function):
    @staticmethod
    def forward(ctx, x):
        return x.clone()

    @staticmethod
    def backward(ctx, g):
        return g.to(torch.bfloat16).double()


def _grad_bf16(x):
    return _GradBf16.apply(x)


def _corrected(U, d):
    """The clipped application of a correction."""
    def thermal(u, faces):
        b = [0.5 * (faces[a] + _next(faces[a], a)) for a in range(3)]
        mag = 0.5 * (b[0] ** 2 + b[1] ** 2 + b[2] ** 2)
        kin = 0.5 * (u[1] ** 2 + u[2] ** 2 + u[3] ** 2) / u[0]
        return u[4] - kin - mag, kin, mag
    floor = 0.5 * thermal(U[:5], U[5:])[0]
    faces = U[5:] + d[5:]
    du = torch.cat([torch.maximum(d[:1], -0.5 * U[:1]), d[1:5]])
    out = U[:5].clone()
    _, kin, mag = thermal(out, faces)
    out[4] = kin + mag + floor
    done = torch.zeros_like(floor, dtype=torch.bool)
    for a in (1.0, 0.5, 0.25, 0.0):
        u = U[:5] + a * du
        ok = (thermal(u, faces)[0] >= floor) & ~done
        out = torch.where(ok, u, out)
        done |= ok
    return torch.cat([out, faces])


def exact(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        return [_advance(s.double(), case["steps"], "ppp", case["floor"]) for _, s in _ensemble_states(case, seed)]
    x = _state(case, seed, torch.float64 if kind == "box64" else torch.float32)
    if kind == "box":
        return _advance(x.double(), case["steps"], case["bc"], case["floor"])
    if kind == "box64":
        return _advance(x, case["steps"])
    U = x.double()
    if kind == "diag":
        div = sum((_next(U[5 + d], d) - U[5 + d]) * U.shape[-1 - d] for d in range(3)).abs().max()
        p, _ = _pressure(U, _centred(U))
        sums = [float(U[q].sum()) for q in range(8)]
        return np.array(sums + [float(div) / max(U.shape[1:]), float(p.min())])
    if kind == "restrict":
        r = case["r"]
        nz, ny, nx = (m // r for m in U.shape[1:])
        blocks = U.view(8, nz, r, ny, r, nx, r)
        out = blocks.mean(dim=(2, 4, 6))
        for d in range(3):  # face fields: the mean over the coarse low face
            out[5 + d] = blocks[5 + d].select(5 - 2 * d, 0).mean(dim=_face_dims(d))
        return out
    norm = _norm(x)
    W, b = _network(seed)
    if kind == "coarse":
        with torch.no_grad():
            d = _correction(x, norm, [w.double() for w in W], [v.double() for v in b], norm.out_scale)
            _step(U, CFL / _rate(U, "ppp"))
            return {"state": _corrected(U, d), "correction": d}
    W = [w.double().requires_grad_() for w in W]
    b = [v.double().requires_grad_() for v in b]
    d = _correction(x, norm, W, b, norm.out_scale)
    weight = torch.tensor(norm.loss_weight, dtype=torch.float32, device="cuda").double().view(8, 1, 1, 1)
    loss = (weight * (d - _target(x, norm, seed).double()) ** 2).sum()
    loss.backward()
    return {"correction": d.detach(), "loss": loss.detach().view(1), "grads": [p.grad for p in (W + b)[:-1]]}


def _face_dims(d):
    """Dimensions to average over in a (nz, r, ny, r, nx, r) field whose sub-cell dimension of axis d was selected away."""
    left = [k for k in (1, 3, 5) if k != 5 - 2 * d]
    return tuple(k if k < 5 - 2 * d else k - 1 for k in left)
