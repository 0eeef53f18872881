"""The work that users of the library have it do, as cases that can be timed and checked.

A case is a dict of plain values; kind says which calls a pass makes:

  fields  olb_init_fields_device, olb_step_async, olb_moments_device on one grid: what a simulation does
          between two outputs, with the fields kept on the device
  resume  olb_set_populations, olb_step_totals, olb_get_populations: a run continued from a checkpoint on
          the host, with its mass and energy recorded, and written back
  sweep   olb_batch_step and olb_batch_moments of every run: a parameter sweep of many small grids
  train   olb_mlp_train: one pass of Adam over a set of stencils (the learned weights)

All inputs come from the seed; sizes and parameters are those of paper_1702_01690_gb300/inputs.py, of the tests
and of the benchmark.  Flows start from a moving fluid (a background velocity, a wave or a few smooth modes), as
runs between two outputs do.
"""
import math

import numpy as np
import torch

from paper_1702_01690_gb300 import inputs, learned, olb

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64 = torch.float64
SIDE_X = {"periodic": 0, "walls": 1, "specular": 2, "half": 3}  # half: specular at x = 0, a wall opposite


# ------------------------------------------------------------------ cases
def _grid(name, nx, ny, steps, field, **more):
    case = {"name": name, "kind": "fields", "nx": nx, "ny": ny, "steps": steps, "field": field, "T0": 1.0,
            "side_x": "periodic", "side_y": "periodic", "precision": 64, "learned": False, "tau": 5e-3, "dt": 0.0}
    case.update(more)
    return case


def listed():
    return [
        # the shear-wave decay of Sec. 6.1 on its own grid: the smallest calls, all launches and latency
        _grid("shear_64x4", 64, 4, 200, "wave", T0=1.1, tau=0.01, dt=0.002),
        # liquid and vapour between two diffuse walls on a strip: one or two tiles per SM
        _grid("planar_1024x8", 1024, 8, 50, "noise", side_x="walls", T0=0.9),
        _grid("planar_1024x8_fp32", 1024, 8, 50, "noise", side_x="walls", T0=0.9, precision=32),
        # the reduced channel (mirror planes and a wall) at a ragged size, continued from a checkpoint
        {**_grid("channel_333x217", 333, 217, 12, "drop", side_x="half", side_y="specular", T0=0.8), "kind": "resume"},
        # a drop in its vapour: the convergence grids of the Laplace test and its full grid
        _grid("laplace_512", 512, 512, 5, "drop", T0=0.9),
        _grid("laplace_2048_fp32", 2048, 2048, 3, "drop", T0=0.9, precision=32),
        # phase separation between cold plates, the benchmark's grid: the largest
        _grid("plates_4096", 4096, 4096, 1, "noise", side_x="walls", T0=0.7),
        _grid("plates_4096_fp32", 4096, 4096, 2, "noise", side_x="walls", T0=0.7, precision=32),
        # the same flow with the learned weights
        _grid("learned_1024", 1024, 1024, 2, "noise", side_x="walls", T0=0.7, learned=True),
        _grid("learned_1024_fp32", 1024, 1024, 2, "noise", side_x="walls", T0=0.7, learned=True, precision=32),
        # a sweep over grid sizes, waves, drops and wall temperatures
        {"name": "sweep_24", "kind": "sweep", "runs": 24, "most": 384, "steps": 8, "precision": 64},
        # training of the weight network, one epoch in minibatches of the default size
        {"name": "train_256k", "kind": "train", "samples": 262144, "batch": 4096},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fields"] * 5 + ["resume", "sweep", "train"])
    if kind == "train":
        return {"kind": kind, "samples": _log(rng, 20000, 400000), "batch": rng.choice([1024, 2048, 4096, 5000, 8192])}
    if kind == "sweep":
        return {"kind": kind, "runs": rng.randint(6, 40), "most": _log(rng, 96, 400), "steps": rng.randint(1, 10),
                "precision": rng.choice([64, 32])}
    side_x = rng.choice(["periodic", "walls", "half", "specular"])
    side_y = "periodic" if side_x in ("periodic", "walls") else rng.choice(["periodic", "specular"])
    nx, ny = _log(rng, 24, 2048), _log(rng, 4, 2048)
    learned_weights = kind == "fields" and rng.random() < 0.25
    if learned_weights:
        side_x, side_y = rng.choice(["walls", "periodic"]), "periodic"
    precision = 64 if kind == "resume" else rng.choice([64, 64, 32])
    # at most about 4 M node-steps in FP64 Jiang-Shu (16.8 M are the largest listed case), 2 M through host memory
    most = 2e6 if kind == "resume" or learned_weights else 4e6
    while nx * ny > most:
        nx, ny = (nx + 1) // 2, (ny + 1) // 2
    steps = max(1, min(100, int(most * rng.uniform(0.3, 1.0) / (nx * ny))))
    # learned weights are for the phase separation they were trained on; on a wave that is uniform along y their
    # guard would decide on rounding noise
    field, T0 = ("noise", 0.7) if learned_weights else rng.choice(
        [("wave", 1.1), ("noise", 0.9), ("noise", 0.7), ("drop", 0.9), ("drop", 0.8)])
    case = _grid("", nx, ny, steps, field, side_x=side_x, side_y=side_y, T0=T0, precision=precision,
                 learned=learned_weights, tau=rng.choice([5e-3, 1e-2]))
    case["kind"] = kind
    del case["name"]
    return case


# ------------------------------------------------------------------ inputs
def _params(case):
    nx, ny = case["nx"], case["ny"]
    ds = 1.0 / max(nx, ny)
    dt = case["dt"] or inputs.stable_dt(ds, n_max=2.2)
    Tw = case["T0"] if case["side_x"] in ("walls", "half") else 1.0
    return inputs.RunParams(nx=nx, ny=ny, ds=ds, dt=dt, tau=case["tau"], Tw=(Tw, Tw), side_x=SIDE_X[case["side_x"]],
                            side_y=2 if case["side_y"] == "specular" else 0)


def _coarse_noise(nx, ny, factor, gen):
    """U(-1, 1) on a grid coarser by factor, Fourier-interpolated (inputs.band_limited_noise on the device)."""
    cy, cx = max(1, ny // factor), max(1, nx // factor)
    r = torch.rand((cy, cx), generator=gen, device=DEV, dtype=F64) * 2 - 1
    if factor == 1:
        return r
    C = torch.fft.fft2(r)
    P = torch.zeros((ny, nx), device=DEV, dtype=torch.complex128)
    hy, hx = (cy + 1) // 2, (cx + 1) // 2
    ly, lx = cy - hy, cx - hx
    P[:hy, :hx] = C[:hy, :hx]
    if lx:
        P[:hy, nx - lx:] = C[:hy, hx:]
    if ly:
        P[ny - ly:, :hx] = C[hy:, :hx]
        if lx:
            P[ny - ly:, nx - lx:] = C[hy:, hx:]
    return torch.fft.ifft2(P).real * ((ny * nx) / (cy * cx))


def _fields(case, p, seed):
    """n, u_x, u_y, T of the case's initial state, [ny][nx] each."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    u = torch.rand(12, generator=gen, device=DEV, dtype=F64).tolist()
    nx, ny = p.nx, p.ny
    X = ((torch.arange(nx, device=DEV, dtype=F64) + 0.5) * p.ds).expand(ny, nx)
    Y = ((torch.arange(ny, device=DEV, dtype=F64) + 0.5) * p.ds).unsqueeze(1).expand(ny, nx)
    Lx, Ly = nx * p.ds, ny * p.ds
    T = torch.full((ny, nx), float(case["T0"] if case["field"] != "noise" else 1.0), device=DEV, dtype=F64)
    two_pi = 2.0 * math.pi
    if case["field"] == "wave":
        # a shear wave carried at a background velocity, uniform along y
        amp = 1e-3 * (0.8 + 0.4 * u[0])
        uy = amp * torch.sin(two_pi * X / Lx + two_pi * u[1])
        return torch.ones_like(T), torch.full_like(T, 0.05 + 0.1 * u[2]), uy.contiguous(), T
    kx, ky = two_pi / Lx, two_pi / Ly
    ux = 1e-3 * torch.sin(kx * X + two_pi * u[3]) * (1.0 + 0.5 * torch.cos(ky * Y + two_pi * u[4]))
    uy = 1e-3 * torch.cos(kx * X + two_pi * u[5]) * (1.0 + 0.5 * torch.sin(ky * Y + two_pi * u[6]))
    if case["field"] == "noise":
        factor = max(1, inputs.noise_factor(nx, p.ds))
        while factor > 1 and ny % factor:
            factor //= 2
        n = 1.0 + 0.01 * _coarse_noise(nx, ny, factor, gen)
    else:
        ng, nl = inputs.MAXWELL[round(case["T0"], 6)]
        R = (0.15 + 0.1 * u[7]) * max(Lx, Ly)
        cx, cy = (0.4 + 0.2 * u[8]) * Lx, (0.4 + 0.2 * u[9]) * Ly
        r = torch.sqrt((X - cx) ** 2 + (Y - cy) ** 2)
        n = ng + 0.5 * (nl - ng) * (1.0 - torch.tanh((r - R) / max(0.02, 3.0 * p.ds)))
    return n.contiguous(), ux.contiguous(), uy.contiguous(), T


def _sweep_runs(case, seed):
    """The runs of a sweep, as inputs.batch_sweep makes them, with amplitudes and phases from the seed."""
    rng = np.random.Generator(np.random.PCG64(seed))
    sizes = [s for s in (32, 48, 64, 96, 128, 192, 256, 384) if s <= case["most"]]
    runs = []
    for r in range(case["runs"]):
        N = sizes[(3 * r) % len(sizes)]
        ds = 1.0 / N
        amp, ph = 1e-3 * rng.uniform(0.8, 1.2), rng.uniform(0, 2 * math.pi)
        if r % 4 < 2:
            p = inputs.RunParams(nx=N, ny=N, ds=ds, dt=inputs.stable_dt(ds), tau=0.01)
            n, ux, uy, T = inputs.shear_wave(N, N, ds, 1.0, 0.8 if r % 8 < 4 else 1.1, 0.0, V=0.05)
            wave = np.tile(amp * np.sin(2 * math.pi * inputs.node_x(N, ds) + ph), (N, 1))
            f = (n, ux + (wave if r % 4 else 0.5 * wave), uy + wave, T)
        elif r % 4 == 2:
            p = inputs.RunParams(nx=N, ny=N, ds=ds, dt=inputs.stable_dt(ds, n_max=1.66), tau=5e-3)
            n, ux, uy, T = inputs.laplace_drop(N, N, ds, 0.15 + 0.15 * rng.random(), 0.9, max(0.02, 3 * ds))
            f = (n, ux + amp, uy + 0.7 * amp, T)
        else:
            Tw = (0.75, 0.8, 0.85, 0.9)[(r // 4) % 4]
            p = inputs.RunParams(nx=2 * N, ny=8, ds=ds / 2, dt=inputs.stable_dt(ds / 2, n_max=2.2), tau=5e-3,
                                 Tw=(Tw, Tw), side_x=1)
            n, ux, uy, T = inputs.cold_rest(2 * N, 8, ds / 2, int(rng.integers(1 << 30)))
            f = (n, ux + amp, uy + 0.7 * amp, T)
        runs.append((p, f))
    return runs


def _stencils(case, seed):
    """Normalised stencils with candidates and targets as learned.harvest gives them: smooth data, steps and kinks."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    S = case["samples"]
    u = torch.rand((S, 6), generator=gen, device=DEV, dtype=F64)
    at = torch.arange(-2, 3, device=DEV, dtype=F64)
    k = 0.2 + 1.6 * u[:, :1]
    step = torch.sigmoid((at - 3.0 + 6.0 * u[:, 4:5]) * (0.5 + 6.0 * u[:, 5:6] ** 2))
    v = torch.sin(k * at + 2 * math.pi * u[:, 1:2]) * u[:, 2:3] + (u[:, 3:4] - 0.5) * step
    half = torch.sin(k * 0.5 + 2 * math.pi * u[:, 1:2]) * u[:, 2:3] + (u[:, 3:4] - 0.5) * torch.sigmoid(
        (0.5 - 3.0 + 6.0 * u[:, 4:5]) * (0.5 + 6.0 * u[:, 5:6] ** 2))
    rng_v = v.max(1, keepdim=True).values - v.min(1, keepdim=True).values + 1e-3
    x = (v - v.mean(1, keepdim=True)) / rng_v
    d = v[:, 1:] - v[:, :-1]
    gn = torch.stack([5 * d[:, 1] - 2 * d[:, 0], d[:, 1] + 2 * d[:, 2], 4 * d[:, 2] - d[:, 3]], 1) / 6 / rng_v
    tn = ((half - v[:, 2:3]) / rng_v)[:, 0]
    return x.float().contiguous(), gn.float().contiguous(), tn.float().contiguous()


def _theta0(seed):
    rng = np.random.default_rng(seed)
    scale = np.concatenate([np.full(160, 0.6), np.zeros(32), np.full(1024, 0.2), np.zeros(32), np.full(96, 0.2),
                            np.zeros(3)])
    return torch.from_numpy((rng.standard_normal(olb.MLP_PARAMS) * scale).astype(np.float32)).to(DEV)


def prepare(case, seed):
    if case["kind"] == "train":
        x, gn, tn = _stencils(case, seed)
        return {"case": case, "x": x, "gn": gn, "tn": tn, "theta": _theta0(seed)}
    if case["kind"] == "sweep":
        runs = _sweep_runs(case, seed)
        b = olb.Batch([p for p, _ in runs], precision=olb.FP64 if case["precision"] == 64 else olb.FP32_KAHAN)
        for r, (_, f) in enumerate(runs):
            b.init_fields(r, *f)
        b.autotune(1)
        return {"case": case, "batch": b}
    p = _params(case)
    fields = _fields(case, p, seed)
    ctx = olb.create(p, precision=olb.FP64 if case["precision"] == 64 else olb.FP32_KAHAN,
                     weno_mode=olb.WENO_LEARNED if case["learned"] else olb.WENO_JS)
    if case["learned"]:
        ctx.set_weno_mlp(learned.load_theta())
    state = {"case": case, "ctx": ctx}
    if case["kind"] == "resume":
        ctx.init_fields(*fields)
        state["f"] = ctx.get_populations()
    else:
        state["fields"] = fields
    return state


# ------------------------------------------------------------------ one pass
def _joined(runs):
    """The fields of all runs of a sweep, one after the other."""
    return {k: np.concatenate([m[q].ravel() for m in runs]) for q, k in enumerate(("n", "ux", "uy", "T"))}


def run(state):
    case = state["case"]
    if case["kind"] == "train":
        theta = state["theta"].clone()
        history = olb.mlp_train(theta, state["x"], state["gn"], state["tn"], epochs=1, batch=case["batch"], lr=1e-3)
        return {"theta": theta, "loss": history}
    if case["kind"] == "sweep":
        b = state["batch"]
        b.step(case["steps"])
        return _joined([b.moments(r) for r in range(b.count)])
    ctx = state["ctx"]
    if case["kind"] == "resume":
        ctx.set_populations(state["f"])
        totals = ctx.step_totals(case["steps"], max(1, case["steps"] // 4))
        return {"f": ctx.get_populations(), "totals": totals}
    ctx.init_fields(*state["fields"])
    ctx.step_async(case["steps"])
    n, ux, uy, T = ctx.moments_device()
    return {"n": n, "ux": ux, "uy": uy, "T": T}


def work(case):
    if case["kind"] == "train":
        # forward and backward of 1280 products per sample, two of them in the backward pass
        return {"bytes": case["samples"] * 36.0, "flops": case["samples"] * 6.0 * 1280}
    if case["kind"] == "sweep":
        nodes = sum(p.nx * p.ny for p, _ in _sweep_runs(case, 0))
    else:
        nodes = case["nx"] * case["ny"]
    # a node and stage: 3571 operations; 50, 75 and 75 population values of 8 bytes in the three stages of a step
    flops, each = 3 * 3571.0, 200 * 8.0
    if case.get("learned"):
        flops += 3 * 40 * 2560.0
    ends = 25 * 16.0 if case["kind"] == "resume" else 32.0 if case["kind"] == "sweep" else 64.0
    return {"bytes": nodes * (each * case["steps"] + ends), "flops": nodes * flops * case["steps"]}


# ------------------------------------------------------------------ the method in 64 bits
_R = [-math.sqrt(5 + math.sqrt(10)), -math.sqrt(5 - math.sqrt(10)), 0.0, math.sqrt(5 - math.sqrt(10)),
      math.sqrt(5 + math.sqrt(10))]
_W = [(7 - 2 * math.sqrt(10)) / 60, (7 + 2 * math.sqrt(10)) / 60, 8 / 15, (7 + 2 * math.sqrt(10)) / 60,
      (7 - 2 * math.sqrt(10)) / 60]


def _he(l, x):
    return (1.0, x, x * x - 1, x ** 3 - 3 * x, x ** 4 - 6 * x * x + 3, x ** 5 - 10 * x ** 3 + 15 * x)[l]


class _Exact:
    """The paper's RK-3 step in 64 bits on [5][5][ny][nx] populations, every equation as it is printed."""

    def __init__(self, p, theta=None):
        self.p = p
        t = lambda v: torch.tensor(v, device=DEV, dtype=F64)  # noqa: E731
        self.R = t(_R)
        self.D = t([[-_W[k] * sum(_he(l + 1, _R[k]) * _he(l, _R[q]) / math.factorial(l) for l in range(4))
                     for q in range(5)] for k in range(5)])
        self.theta = None if theta is None else torch.as_tensor(theta, device=DEV).to(F64)
        ar = lambda n: torch.arange(-3, n + 3, device=DEV)  # noqa: E731

        def mirrored(n, lo, hi):
            i = ar(n)
            wrapped = i % n
            i = torch.where(i < 0, -1 - i if lo else wrapped, i)
            return torch.where(ar(n) >= n, 2 * n - 1 - ar(n) if hi else wrapped, i)

        self.ix = mirrored(p.nx, p.side_x in (1, 2, 3), p.side_x in (1, 2, 3))
        self.iy = mirrored(p.ny, p.side_y == 2, p.side_y == 2)
        w = {(1, 0): 31 / 70, (0, 1): 31 / 70, (1, 1): 27 / 140, (2, 1): -3 / 70, (1, 2): -3 / 70, (2, 2): 3 / 560,
             (3, 0): -1 / 630, (0, 3): -1 / 630, (3, 1): 1 / 280, (1, 3): 1 / 280}
        c = {(3, 3): -17 / 2160, (0, 3): -59 / 540, (2, 2): 13 / 120, (1, 2): -7 / 30, (0, 2): 5 / 4, (2, 1): -7 / 60,
             (1, 1): 187 / 240, (0, 1): -59 / 20}
        both = [(l, m) for l in (-3, -2, -1, 1, 2, 3) for m in range(-3, 4)]
        self.grad = {(l, m): l * w[abs(l), abs(m)] for l, m in both if (abs(l), abs(m)) in w}
        self.glap = {(l, m): math.copysign(1, l) * c[abs(m), abs(l)] for l, m in both if (abs(m), abs(l)) in c}

    def g(self, u, T):
        """The factors g_k(u, T) of the equilibrium, [5] + u.shape."""
        th = T - 1
        c = [torch.ones_like(u), u, 0.5 * (u * u + th), u ** 3 / 6 + 0.5 * th * u,
             u ** 4 / 24 + 0.25 * th * u * u + 0.125 * th * th]
        return torch.stack([_W[k] * sum(_he(l, _R[k]) * c[l] for l in range(5)) for k in range(5)])

    def feq(self, n, ux, uy, T):
        return n * self.g(ux, T)[:, None] * self.g(uy, T)[None]

    def moments(self, f):
        n = f.sum((0, 1))
        fx, fy = f.sum(1), f.sum(0)
        R = self.R.view(5, 1, 1)
        ux, uy = (R * fx).sum(0) / n, (R * fy).sum(0) / n
        return n, ux, uy, 0.5 * ((R * R * (fx + fy)).sum(0) / n - ux * ux - uy * uy)

    def weno(self, v):
        d = [v[q + 1] - v[q] for q in range(4)]
        s1 = 13 / 12 * (d[1] - d[0]) ** 2 + 0.25 * (3 * d[1] - d[0]) ** 2
        s2 = 13 / 12 * (d[2] - d[1]) ** 2 + 0.25 * (d[1] + d[2]) ** 2
        s3 = 13 / 12 * (d[3] - d[2]) ** 2 + 0.25 * (3 * d[2] - d[3]) ** 2
        F1, F2, F3 = (5 * d[1] - 2 * d[0]) / 6, (d[1] + 2 * d[2]) / 6, (4 * d[2] - d[3]) / 6
        low = torch.minimum(s1, torch.minimum(s2, s3))
        zero = low == 0
        w1, w2, w3 = [torch.where(zero, g * (s == 0), g * (low / s) ** 2) for g, s in ((0.1, s1), (0.6, s2), (0.3, s3))]
        js = (w1 * F1 + w2 * F2 + w3 * F3) / (w1 + w2 + w3)
        if self.theta is not None:
            high = torch.maximum(s1, torch.maximum(s2, s3))
            acts = ~zero & (low < 0.9 * high)
            x = torch.stack([q[acts] for q in v], -1)
            if x.numel():
                span = x.max(-1, keepdim=True).values - x.min(-1, keepdim=True).values
                w = _net(self.theta, (x - x.mean(-1, keepdim=True)) / span)
                js[acts] = w[:, 0] * F1[acts] + w[:, 1] * F2[acts] + w[:, 2] * F3[acts]
        return v[2] + js

    def wall(self, f, hi):
        """Ghost layers 0, 1, 2 of a diffuse wall, [3][5][5][ny]."""
        p, s = self.p, 1 if hi else 0
        a = [f[..., -1 - q] if hi else f[..., q] for q in range(3)]
        out = slice(3, 5) if hi else slice(0, 2)
        inc = slice(0, 2) if hi else slice(3, 5)
        G = torch.zeros((3,) + a[0].shape, device=DEV, dtype=F64)
        G[0, out] = (3 * a[0] - 3 * a[1] + a[2])[out]
        G[1, out] = (6 * a[0] - 8 * a[1] + 3 * a[2])[out]
        flux = self.R[out].view(2, 1, 1) * self.weno([a[2][out], a[1][out], a[0][out], G[0, out], G[1, out]])
        one = torch.ones(1, device=DEV, dtype=F64)
        geq = (self.g(0 * one, p.Tw[s] * one)[:, None] * self.g(p.uw[s] * one, p.Tw[s] * one)[None])[..., 0]
        nw = -flux.sum((0, 1)) / (geq[inc] * self.R[inc].view(2, 1)).sum()
        G[:, inc] = (nw * geq[inc].unsqueeze(-1)).unsqueeze(0)
        return G

    def L(self, f):
        p = self.p
        n, ux, uy, T = self.moments(f)
        dp = n * T - (n * T / (1 - p.b * n) - p.a * n * n)
        E = lambda a: a[self.iy][:, self.ix]  # noqa: E731
        ndp, nn = E(dp), E(n)

        def stencil(a, c, along_x):
            acc = torch.zeros_like(n)
            for (l, m), w in c.items():
                i, j = (l, m) if along_x else (m, l)
                acc += w * a[3 + j:3 + j + p.ny, 3 + i:3 + i + p.nx]
            return acc

        Fx = stencil(ndp, self.grad, True) / p.ds / n + p.sigma * stencil(nn, self.glap, True) / p.ds ** 3
        Fy = stencil(ndp, self.grad, False) / p.ds / n + p.sigma * stencil(nn, self.glap, False) / p.ds ** 3
        L = (self.feq(n, ux, uy, T) - f) / p.tau
        for k in range(5):
            for q in range(5):
                if float(self.D[k, q]) != 0.0:
                    L[k] -= self.D[k, q] * Fx * f[q]
                    L[:, k] -= self.D[k, q] * Fy * f[:, q]
        del Fx, Fy, ndp, nn, dp
        # x faces: extended rows of the populations, walls and mirror planes in the ghost columns
        walls = [self.wall(f, hi) if p.side_x == 1 or (p.side_x == 3 and hi) else None for hi in (False, True)]
        for ks in (slice(0, 2), slice(3, 5)):
            e = f[ks][..., self.ix]
            m = f.flip(0)[ks]
            if p.side_x in (2, 3):
                e[..., :3] = m[..., self.ix[:3]]
            if p.side_x == 2:
                e[..., -3:] = m[..., self.ix[-3:]]
            for hi in (False, True):
                if walls[hi] is not None:
                    for q in range(3):
                        e[..., (p.nx + 3 + q) if hi else 2 - q] = walls[hi][q][ks]
            at = [q if ks.start else 5 - q for q in range(5)]
            F = self.weno([e[..., q:q + p.nx + 1] for q in at])
            L[ks] -= self.R[ks].view(2, 1, 1, 1) * (F[..., 1:] - F[..., :-1]) / p.ds
            del e, F
        for ks in (slice(0, 2), slice(3, 5)):
            e = f[:, ks][..., self.iy, :]
            if p.side_y == 2:
                m = f.flip(1)[:, ks]
                e[..., :3, :] = m[..., self.iy[:3], :]
                e[..., -3:, :] = m[..., self.iy[-3:], :]
            at = [q if ks.start else 5 - q for q in range(5)]
            F = self.weno([e[..., q:q + p.ny + 1, :] for q in at])
            L[:, ks] -= self.R[ks].view(1, 2, 1, 1) * (F[..., 1:, :] - F[..., :-1, :]) / p.ds
            del e, F
        return L

    def step(self, f):
        dt = self.p.dt
        f1 = f + dt * self.L(f)
        f2 = 0.75 * f + 0.25 * f1 + 0.25 * dt * self.L(f1)
        del f1
        return f / 3 + 2 / 3 * f2 + 2 / 3 * dt * self.L(f2)


def _net(th, x):
    W1, b1, W2, b2, W3, b3 = torch.split(th, [160, 32, 1024, 32, 96, 3])
    h = torch.tanh(x @ W1.view(32, 5).T + b1)
    return torch.softmax(torch.tanh(h @ W2.view(32, 32).T + b2) @ W3.view(3, 32).T + b3, -1)


def _exact_train(case, seed):
    x, gn, tn = (v.to(F64) for v in _stencils(case, seed))
    th = _theta0(seed).to(F64)
    m, v = torch.zeros_like(th), torch.zeros_like(th)
    S, B, losses = case["samples"], case["batch"], []
    for step, off in enumerate(range(0, S, B), 1):
        t = th.clone().requires_grad_()
        loss = ((_net(t, x[off:off + B]) * gn[off:off + B]).sum(1) - tn[off:off + B]).square().mean()
        (g,) = torch.autograd.grad(loss, t)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        th = th - 1e-3 * (m / (1 - 0.9 ** step)) / ((v / (1 - 0.999 ** step)).sqrt() + 1e-8)
        losses.append(float(loss.detach()))
    return {"theta": th, "loss": np.array([sum(losses) / len(losses)])}


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "sweep":
        out = []
        for p, f in _sweep_runs(case, seed):
            o = _Exact(p)
            f = o.feq(*[torch.from_numpy(np.ascontiguousarray(v)).to(DEV) for v in f])
            for _ in range(case["steps"]):
                f = o.step(f)
            out.append([v.cpu().numpy() for v in o.moments(f)])
        return _joined(out)
    p = _params(case)
    o = _Exact(p, learned.load_theta() if case["learned"] else None)
    f = o.feq(*_fields(case, p, seed))
    every, totals = max(1, case["steps"] // 4), []
    for k in range(case["steps"]):
        f = o.step(f)
        if (k + 1) % every == 0 and case["kind"] == "resume":
            n, ux, uy, T = o.moments(f)
            e = 0.5 * (2 * n * T + n * (ux * ux + uy * uy))
            totals.append([float(q.sum()) * p.ds ** 2 for q in (n, n * ux, n * uy, e)])
    if case["kind"] == "resume":
        return {"f": f.reshape(25, p.ny, p.nx), "totals": np.array(totals)}
    n, ux, uy, T = o.moments(f)
    return {"n": n, "ux": ux, "uy": uy, "T": T}
