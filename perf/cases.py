"""Performance cases of the nlM lattice-Boltzmann library: what its users run, through its public calls.

A case is a dict of plain values.  ``listed()`` gives the fixed ones, ``draw(rng)`` more of the same
ranges; ``prepare`` builds the handles and buffers a user's program keeps, ``run`` is one pass of that
program, ``work`` the bytes and operations the pass cannot do without, and ``exact`` the same results
in 64-bit torch, written from the scheme's equations.  Kinds of case:

  channel    one channel from a seeded density perturbation: a run of steps, then the fields
  transient  the run-control loop: body force set, one step, flux / max |u| read back, every step
  sweep      many uneven 4-column channels in the persistent batched launch (lb_run_until_steady)
  train      the surrogate's training: Adam steps on mini-batches, loss and weights read back
  warmstart  the surrogate's use: network outputs for a batch of channels, start states written

Every handle lives on the current stream; prepared states start from the seed alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1310_7450_gb300 import lbnlm

# ---- the cases -------------------------------------------------------------------------------


def _channel(name, nx, ny, precision, steps, **kw):
    c = dict(name=name, kind="channel", nx=nx, ny=ny, precision=precision, steps=steps, x_mode="periodic",
             walls="bounce_back", stress_mode=0, relaxation=False, stochastic=False)
    c.update(kw)
    return c


def listed():
    return [
        # the parity channel of the oracle runs (4 x 64, theta = 100, FP64): launches and latency
        _channel("oracle_4x64_f64", 4, 64, "f64", 200),
        # the paper's grid, 400 nodes across and 20 along the channel: a small production run
        _channel("paper_20x400_f32", 20, 400, "f32", 200),
        # planar Couette start-up in FP64 (flow curves, reference profiles), odd height
        _channel("couette_256x257_f64", 256, 257, "f64", 16, walls="couette"),
        # a channel whose sides are no multiples of anything
        _channel("ragged_1000x777_f32", 1000, 777, "f32", 16),
        # the single large channel of the benchmark, stress stored every step
        _channel("large_4096x4096_f32", 4096, 4096, "f32", 16),
        # reduced-precision storage on its own channel shape
        _channel("large_8192x2048_bf16", 8192, 2048, "bf16", 16),
        # pressure-driven ends (generalized periodic boundaries)
        _channel("gpbc_2048x1000_f32", 2048, 1000, "f32", 16, x_mode="gpbc"),
        # integral model: carried stress, density-dependent Maxwell time and fluidity memory
        _channel("memory_2048x1024_f32", 2048, 1024, "f32", 16, stress_mode=1, relaxation=True),
        # start-up / cessation control loop on a channel of ordinary size
        dict(name="transient_1024x1024_f32", kind="transient", nx=1024, ny=1024, precision="f32", steps=16),
        # the parameter sweep: uneven channels from rest in one persistent launch
        dict(name="sweep_128_f32", kind="sweep", channels=128, precision="f32", check=500, steps=2000, ny_lo=32,
             ny_hi=1024),
        # eight Adam steps of the 4 -> 256 -> 256 -> 768 surrogate, then its weights
        dict(name="train_256", kind="train", batch=256, steps=8),
        # 512 held-out channels: prediction, decoded start states, their fields
        dict(name="warmstart_512", kind="warmstart", channels=512, ny_lo=32, ny_hi=1024),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "small", "wide", "wide", "wide", "wide", "transient", "sweep", "train", "warmstart"])
    if kind == "small":  # narrow channels: the oracle's and the paper's grids
        nx, ny = _logint(rng, 3, 40), _logint(rng, 24, 600)
        prec = rng.choice(["f64", "f32"])
        walls = rng.choice(["bounce_back", "bounce_back", "couette"])
        return {k: v for k, v in _channel("", nx, ny, prec, _logint(rng, 40, 400), walls=walls).items() if k != "name"}
    if kind == "wide":  # from a few strips to the benchmark's size; half of the widths are ragged
        prec = rng.choice(["f32", "f32", "f32", "bf16", "bf16", "f64"])
        top = 1 << (17 if prec == "f64" else 23)
        while True:
            nx, ny = _logint(rng, 100, 8192), _logint(rng, 33, 4096)
            if rng.random() < 0.5:
                nx = max(128, (nx + 64) // 128 * 128)
            if nx * ny <= top:
                break
        opt = rng.choice(["plain", "plain", "plain", "gpbc", "couette", "mode1", "memory", "stochastic"])
        kw = dict(x_mode="gpbc" if opt == "gpbc" else "periodic", walls="couette" if opt == "couette" else "bounce_back",
                  stress_mode=1 if opt in ("mode1", "memory") else 0, relaxation=opt == "memory",
                  stochastic=opt == "stochastic" and prec == "bf16")
        return {k: v for k, v in _channel("", nx, ny, prec, _logint(rng, 4, 24), **kw).items() if k != "name"}
    if kind == "transient":
        return dict(kind="transient", nx=_logint(rng, 64, 2048), ny=_logint(rng, 64, 2048),
                    precision=rng.choice(["f32", "bf16"]), steps=_logint(rng, 8, 32))
    if kind == "sweep":
        return dict(kind="sweep", channels=_logint(rng, 8, 200), precision="f32", check=500,
                    steps=500 * rng.randint(2, 4), ny_lo=32, ny_hi=_logint(rng, 100, 1024))
    if kind == "train":
        return dict(kind="train", batch=_logint(rng, 24, 512), steps=rng.randint(2, 8))
    return dict(kind="warmstart", channels=_logint(rng, 16, 512), ny_lo=32, ny_hi=_logint(rng, 200, 1024))


# ---- inputs ----------------------------------------------------------------------------------
# Perturbation of the starting density: large enough that every node carries resolved gradients.
AMP = 1e-3
U_WALL = 0.02
RELAX = (2.0, 1.0, 50.0)  # beta_rho, rho_ref, tau_f
H, N_IN, N_OUT, GRID = 256, 4, 768, 256  # surrogate: width, inputs, outputs; points per field
LR = 1e-3


def _params(c, seed):
    """Lattice parameters of a single channel: tau_LB = 0.9, gamma_c = 0.1, theta = 100, with eta^N
    matched to the low-shear viscosity.  Narrow channels take the yield-stress recipe (w_p H = 1/2 at a
    fixed peak speed), wide ones the benchmark's modulus; the force keeps long runs below |u| = 0.1."""
    nu, theta, ny = 0.4 / 3.0, 100.0, c["ny"]
    if c["nx"] <= 64:
        g = 2.0627e-7 * (64.0 / ny) ** 2
        G = g * ny  # w_p H = g H / G = 1/2
    else:
        g = 1e-6 if ny > 2048 else 1e-6 * min(1.0, (256.0 / ny) ** 2)
        G = 1e-3
    return dict(tau_lb=0.9, g_x=g, G_inf=G, tau0=nu / (G * (1.0 + theta)), theta=theta, gamma_c=0.1, rho0=1.0,
                rho_pert_amp=AMP, seed=int(seed) + 1)


def _sweep_params(n, ny_lo, ny_hi, seed):
    """The sweep's draws: Ny uniform, b log-uniform in [1e-8, 1e-5] with g = b (32/Ny)^2, theta =
    10^(2 + 10 eps), eps uniform in [-0.1, 0.1]; G_inf the smallest >= 1e-6 whose steady peak speed is
    at most 0.05 (bisection in log G, all channels at once)."""
    ny = np.random.default_rng(n).integers(ny_lo, ny_hi + 1, n)  # (one grid per case, whatever the seed)
    r = np.random.default_rng(int(seed) + 17)
    g = 10.0 ** r.uniform(-8.0, -5.0, n) * (32.0 / ny) ** 2
    theta = 10.0 ** (2.0 + 10.0 * r.uniform(-0.1, 0.1, n))
    nu, gc, d = 0.4 / 3.0, 0.1, np.linspace(0.0, 1.0, 401)[None, :]

    def peak(logG):
        G = np.exp(logG)
        tau0 = nu / (G * (1.0 + theta))
        w = (g * ny / 2.0 / G)[:, None] * d
        b = (gc * (1.0 + theta) / (2.0 * theta))[:, None]
        dv = -w / 2.0 + b - np.sqrt((w / 2.0 - b) ** 2 + w * (gc / theta)[:, None])
        return -(dv[:, 1:] + dv[:, :-1]).sum(1) / 800.0 * ny / 2.0 / tau0

    lo, hi = np.full(n, math.log(1e-6)), np.zeros(n)
    over = peak(lo) > 0.05
    for _ in range(40):
        mid = 0.5 * (lo + hi)
        up = peak(mid) > 0.05
        lo, hi = np.where(up, mid, lo), np.where(up, hi, mid)
    G = np.where(over, np.exp(hi), 1e-6)
    return [dict(ny=int(ny[k]), tau_lb=0.9, g_x=float(g[k]), G_inf=float(G[k]),
                 tau0=float(nu / (G[k] * (1.0 + theta[k]))), theta=float(theta[k]), gamma_c=gc, rho0=1.0)
            for k in range(n)]


def _drive(p, k, n):
    """Body force of step k of a transient: one period of a 50 % modulation over the n steps."""
    return p["g_x"] * (1.0 + 0.5 * math.cos(2.0 * math.pi * k / n))


def _weights(seed):
    """Surrogate weights, flat in the library's order: uniform in +-1/sqrt(fan in), small biases."""
    g = torch.Generator().manual_seed(int(seed) + 5)
    parts = []
    for o, i in ((H, N_IN), (H, H), (N_OUT, H)):
        parts.append(((torch.rand(o, i, generator=g) * 2 - 1) / math.sqrt(i)).reshape(-1))
        parts.append((torch.rand(o, generator=g) * 2 - 1) * 0.1)
    return torch.cat(parts)


def _batches(c, seed):
    """Standardised features and targets of `steps` mini-batches (smooth functions of the features)."""
    g = torch.Generator().manual_seed(int(seed) + 9)
    x = torch.randn(c["steps"], c["batch"], N_IN, generator=g)
    phase = torch.rand(N_OUT, generator=g) * 6.0
    mix = torch.randn(N_IN, N_OUT, generator=g) * 0.7
    return x.contiguous(), torch.sin(x @ mix + phase).contiguous()


def _features(ps):
    x = np.array([[math.log10(p["ny"]), math.log10(p["g_x"]), math.log10(p["G_inf"]), math.log10(p["theta"])] for p in ps])
    return torch.tensor((x - x.mean(0)) / (x.std(0) + 1e-12), dtype=torch.float32).contiguous()


def _standardisation(seed):
    g = torch.Generator().manual_seed(int(seed) + 13)
    return 0.01 * torch.randn(N_OUT, generator=g), 0.01 + 0.02 * torch.rand(N_OUT, generator=g)


class _State:
    """What a user's program keeps; handles are given back when it goes."""

    sim = mlp = None

    def __del__(self):
        if self.sim is not None:
            self.sim.close()
        if self.mlp is not None:
            lbnlm.lb_mlp_destroy(self.mlp)


def _field_buffers(s, precision, sigma=True):
    dt = torch.float64 if precision == "f64" else torch.float32
    s.code = 0 if precision == "f64" else 1
    n = s.sim.nodes
    s.u = torch.empty(n, 2, dtype=dt, device="cuda")
    s.sigma = torch.empty(n, 4, dtype=dt, device="cuda") if sigma else None
    s.rho = torch.empty(n, dtype=dt, device="cuda")


def _flags(c):
    f = lbnlm.LB_GRID_STORE_SIGMA
    if c.get("stochastic"):
        f |= lbnlm.LB_GRID_BF16_STOCHASTIC
    if c.get("relaxation"):
        f |= lbnlm.LB_GRID_RELAXATION_MODEL
    return f


def prepare(case, seed):
    s = _State()
    s.case = case
    stream = torch.cuda.current_stream().cuda_stream
    kind = case["kind"]
    if kind == "channel":
        s.sim = lbnlm.Channels(case["nx"], case["ny"], _params(case, seed), case["precision"],
                               stress_mode=case["stress_mode"], flags=_flags(case), stream=stream,
                               x_mode=case["x_mode"], walls=case["walls"])
        if case["relaxation"]:
            lbnlm.lb_set_relaxation_model(s.sim.h, -1, *RELAX)
        if case["walls"] == "couette":
            lbnlm.lb_set_wall_velocity(s.sim.h, -1, U_WALL)
        _field_buffers(s, case["precision"])
    elif kind == "transient":
        s.p = _params(case, seed)
        s.sim = lbnlm.Channels(case["nx"], case["ny"], s.p, case["precision"], flags=_flags(case), stream=stream)
        lbnlm.lb_set_monitor_mode(s.sim.h, lbnlm.LB_MONITOR_FLUX_MAX)
        s.mon = torch.zeros(case["steps"], 4, dtype=torch.float64, device="cuda")
        s.rows = [s.mon[k] for k in range(case["steps"])]
        _field_buffers(s, case["precision"])
    elif kind == "sweep":
        ps = _sweep_params(case["channels"], case["ny_lo"], case["ny_hi"], seed)
        s.sim = lbnlm.Channels(4, [p["ny"] for p in ps], ps, case["precision"], stream=stream)
        lbnlm.lb_sweep_tune(s.sim.h)
        _field_buffers(s, case["precision"])
    elif kind == "train":
        s.mlp = lbnlm.lb_mlp_create(N_IN, H, N_OUT, case["batch"], 0, stream)
        lbnlm.lb_mlp_set_params(s.mlp, _weights(seed).numpy())
        x, y = _batches(case, seed)
        s.x, s.y = x.cuda(), y.cuda()
        s.params = np.zeros(lbnlm.lb_mlp_num_params(s.mlp), dtype=np.float32)
    else:
        ps = _sweep_params(case["channels"], case["ny_lo"], case["ny_hi"], seed)
        s.sim = lbnlm.Channels(4, [p["ny"] for p in ps], ps, "f32", stream=stream)
        s.mlp = lbnlm.lb_mlp_create(N_IN, H, N_OUT, case["channels"], 0, stream)
        lbnlm.lb_mlp_set_params(s.mlp, _weights(seed).numpy())
        s.x = _features(ps).cuda()
        s.mu, s.sd = (t.cuda() for t in _standardisation(seed))
        s.pred = torch.empty(case["channels"], N_OUT, dtype=torch.float32, device="cuda")
        _field_buffers(s, "f32", sigma=False)
    return s


def _fields(s):
    lbnlm.lb_get_fields(s.sim.h, s.u, s.sigma, s.rho, s.code, True)


def run(state):
    s, c = state, state.case
    kind = c["kind"]
    if kind == "channel":
        s.sim.step(c["steps"])
        _fields(s)
        return {"u": s.u, "sigma": s.sigma, "rho": s.rho}
    if kind == "transient":
        h, n = s.sim.h, c["steps"]
        for k in range(n):
            lbnlm.lb_set_body_force(h, -1, _drive(s.p, k, n))
            lbnlm.lb_step(h, 1)
            lbnlm.lb_monitor_async(h, s.rows[k])
        _fields(s)
        return {"u": s.u, "sigma": s.sigma, "rho": s.rho, "flux_max": s.mon[:, 1:3].float()}
    if kind == "sweep":
        steps, _ = s.sim.run_until_steady(1e-30, c["check"], c["steps"])
        _fields(s)
        return {"u": s.u, "sigma": s.sigma, "rho": s.rho, "steps": steps}
    if kind == "train":
        n = c["steps"]
        for k in range(n):
            loss = lbnlm.lb_mlp_train_step(s.mlp, s.x[k], s.y[k], c["batch"], LR, want_loss=k == n - 1)
        lbnlm.lb_mlp_get_params(s.mlp, s.params)
        return {"params": s.params, "loss": np.float32(loss)}
    lbnlm.lb_mlp_forward(s.mlp, s.x, c["channels"], s.pred)
    lbnlm.lb_warmstart_apply(s.sim.h, s.pred, s.mu, s.sd)
    _fields(s)
    return {"pred": s.pred, "u": s.u, "rho": s.rho}


# ---- work ------------------------------------------------------------------------------------

STEP_FLOPS = 220  # one node, one step: moments, gradients, 2 x 2 stress solve, collision
FIELD_FLOPS = 100


def work(case):
    kind = case["kind"]
    if kind in ("channel", "transient"):
        t, a = {"f64": (8, 8), "f32": (4, 4), "bf16": (2, 4)}[case["precision"]]
        n = case["nx"] * case["ny"]
        state = 9 * t + a + (3 * a if case.get("stress_mode") else 0) + (8 if case.get("relaxation") else 0)
        fields = n * (state + 7 * a)
        # a state that fits the chip's caches crosses memory once per pass, a larger one every step
        passes = case["steps"] if 2 * 9 * t * n > 120e6 else 1
        return {"bytes": n * passes * (2 * state + 3 * a) + fields,
                "flops": n * (case["steps"] * STEP_FLOPS + FIELD_FLOPS)}
    if kind == "train":
        w = H * N_IN + H * H + N_OUT * H + 2 * H + N_OUT
        b = case["batch"]
        fwd = H * N_IN + H * H + N_OUT * H
        return {"bytes": case["steps"] * (b * (N_IN + N_OUT) * 4 + 6 * 4 * w) + 4 * w,
                "flops": case["steps"] * 2 * b * (3 * fwd - H * N_IN)}
    n = 4 * sum(p["ny"] for p in _sweep_params(case["channels"], case["ny_lo"], case["ny_hi"], 0))
    if kind == "sweep":
        return {"bytes": n * (2 * 40 + 40 + 28), "flops": n * (case["steps"] * STEP_FLOPS + FIELD_FLOPS)}
    w, b = H * N_IN + H * H + N_OUT * H, case["channels"]
    return {"bytes": n * (40 + 40 + 12) + 2 * w + b * (N_IN + N_OUT) * 4, "flops": 2 * b * w + n * FIELD_FLOPS}


# ---- the same in 64 bits ---------------------------------------------------------------------
# D2Q9: rest, +x, +y, -x, -y, and the diagonals.  All channels' rows are stacked along dim 0;
# `first` / `last` mark the wall rows, and parameters are one column per row.
CX, CY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


def _uniform(seed, n):
    """U(-1, 1) of SplitMix64 outputs 1 .. n."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + np.arange(1, n + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return (z >> np.uint64(11)).astype(np.float64) * 2.0 ** -52 - 1.0


class _Exact:
    """The scheme of the library's header on deviations d_i = n_i - w_i, in float64 torch."""

    def __init__(self, nx, nys, ps, x_mode="periodic", walls="bounce_back", stress_mode=0, relax=None, u_wall=0.0):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        rep = torch.tensor(nys, device=dev)

        def col(f):
            v = torch.tensor([f(p) for p in ps], dtype=torch.float64, device=dev)
            return v if len(ps) == 1 else torch.repeat_interleave(v, rep)[:, None]

        self.nx, self.rows, self.dev = nx, sum(nys), dev
        ends = torch.cumsum(rep, 0)
        idx = torch.arange(self.rows, device=dev)
        self.first = torch.isin(idx, ends - rep)[:, None]
        self.last = torch.isin(idx, ends - 1)[:, None]
        self.gpbc, self.couette, self.mode, self.relax, self.u_wall = x_mode == "gpbc", walls == "couette", stress_mode, relax, u_wall
        self.om = 1 / 0.9
        self.k2 = 1 - 0.5 * self.om
        self.k1 = -4.5 * self.om
        self.kdr = 0.0 if self.gpbc else 1.0
        self.g = col(lambda p: 0.0 if self.gpbc else p["g_x"])
        self.G, self.tau = col(lambda p: p["G_inf"]), col(lambda p: p["theta"] * p["tau0"])
        self.igc = col(lambda p: 1 / p["gamma_c"])
        self.cD = col(lambda p: p["G_inf"] * p["tau0"] - 0.4 / 3)
        half = 1.5 * ps[0]["g_x"] * (nx + 1)
        self.rho_in, self.rho_out = half, -half
        z = lambda: torch.zeros(self.rows, nx, dtype=torch.float64, device=dev)  # noqa: E731
        self.drho, self.phi = z(), z()
        self.sig = [z(), z(), z()] if stress_mode else None
        self.d = None

    def start(self, seed, amp):
        rho = (1.0 + amp * torch.from_numpy(_uniform(seed, self.rows * self.nx))).reshape(self.rows, self.nx).to(self.dev) - 1.0
        if self.gpbc:
            x = torch.arange(self.nx, dtype=torch.float64, device=self.dev)
            rho = rho + self.rho_in + (self.rho_out - self.rho_in) * (x + 1) / (self.nx + 1)
        self.d = torch.stack([w * rho for w in W])

    def _pull(self):
        d, out = self.d, []
        if self.gpbc:
            def shift(col, delta, i):
                s = d[:, :, col]
                jx, jy = s[1] - s[3] + s[5] - s[6] - s[7] + s[8], s[2] - s[4] + s[5] + s[6] - s[7] - s[8]
                r, cj = 1 + s.sum(0), CX[i] * jx + CY[i] * jy
                dl = delta - s.sum(0).mean()
                return W[i] * (dl - (4.5 * cj * cj - 1.5 * (jx * jx + jy * jy)) * dl / (r * (r + dl)))
        for i in range(9):
            src = d[i]
            if self.gpbc and CX[i]:
                src = src.clone()
                col, delta = (self.nx - 1, self.rho_in) if CX[i] == 1 else (0, self.rho_out)
                src[:, col] += shift(col, delta, i)
            v = torch.roll(src, (CY[i], CX[i]), (0, 1)) if CX[i] or CY[i] else src
            if CY[i]:
                v = torch.where(self.first if CY[i] == 1 else self.last, d[OPP[i]], v)
            out.append(v)
        if self.couette:
            uw, top = self.u_wall, -1
            r = 1 + out[0][top] + out[1][top] + out[3][top] + 2 * (out[2][top] + out[5][top] + out[6][top])
            ht = 0.5 * (out[1][top] - out[3][top])
            out[4], out[7], out[8] = out[4].clone(), out[7].clone(), out[8].clone()
            out[4][top] = out[2][top]
            out[7][top] = out[5][top] + ht - 0.5 * r * uw
            out[8][top] = out[6][top] - ht + 0.5 * r * uw
        return out

    def _ddy(self, f):
        up, dn = torch.roll(f, -1, 0), torch.roll(f, 1, 0)
        v = 0.5 * (up - dn)
        v = torch.where(self.first, 0.5 * (-3 * f + 4 * up - torch.roll(f, -2, 0)), v)
        return torch.where(self.last, 0.5 * (3 * f - 4 * dn + torch.roll(f, 2, 0)), v)

    def _state(self):
        """Everything of one step up to the collision."""
        n = self._pull()
        dR = sum(n[1:], n[0])
        jx = n[1] - n[3] + n[5] - n[6] - n[7] + n[8] + 0.5 * self.g
        jy = n[2] - n[4] + n[5] + n[6] - n[7] - n[8]
        ux, uy = jx / (1 + dR), jy / (1 + dR)
        a, c = (0.5 * (torch.roll(f, -1, 1) - torch.roll(f, 1, 1)) for f in (ux, uy))
        b, e = self._ddy(ux), self._ddy(uy)
        Dxx, Dxy, Dyy = 2 * a, b + c, 2 * e
        sII = torch.sqrt(0.5 * (Dxx * Dxx + 2 * Dxy * Dxy + Dyy * Dyy))
        phi = self.phi
        if self.relax:
            beta, ref, tf = self.relax
            tau = self.tau * torch.exp(beta * (1 + dR - self.drho - ref) / ref)
            ss = 1 / tau + sII * self.igc
            phi = torch.where(phi > 0, (tf * phi + ss) / (tf + 1), ss) if tf > 0 else phi
            tm = 1 / phi if tf > 0 else 1 / ss
        else:
            tm = self.tau / (1 + self.tau * sII * self.igc)
        # s - al (kappa s + s kappa^T) = rhs, as three equations for (xx, xy, yy)
        if self.mode:
            al = tm / (tm + 1)
            r1, r2, r3 = (al * (s + self.G * D) for s, D in zip(self.sig, (Dxx, Dxy, Dyy)))
        else:
            al = tm
            r1, r2, r3 = (self.G * tm * D for D in (Dxx, Dxy, Dyy))
        A, E, Pq = 1 - 2 * al * a, 1 - 2 * al * e, 1 - al * (a + e)
        # xx = (r1 + 2 al b xy)/A, yy = (r3 + 2 al c xy)/E, and xy from the middle equation
        xy = (r2 + al * c * r1 / A + al * b * r3 / E) / (Pq - 2 * al * al * b * c * (1 / A + 1 / E))
        xx, yy = (r1 + 2 * al * b * xy) / A, (r3 + 2 * al * c * xy) / E
        N = (xx + self.cD * Dxx, xy + self.cD * Dxy, yy + self.cD * Dyy)
        drho = self.kdr * -1.5 * (N[0] + N[2])
        S = drho - self.kdr * self.drho
        req = dR + 0.5 * S
        return n, jx, jy, (xx, xy, yy), N, drho, S, req, phi

    def fields(self):
        _, jx, jy, s, _, drho, _, req, _ = self._state()
        rho = 1 + req - drho
        u = torch.stack([jx / rho, jy / rho], -1).reshape(-1, 2)
        sig = torch.stack([s[0], s[2], torch.zeros_like(s[0]), s[1]], -1).reshape(-1, 4)
        return u, sig, rho.reshape(-1)

    def step(self):
        """One step; returns (flux, max |u|) of the state it starts from."""
        n, jx, jy, s, N, drho, S, req, phi = self._state()
        rq, g, om, k2 = 1 + req, self.g, self.om, self.k2
        ux, uy = jx / rq, jy / rq
        Yxx, Yyy, Yxy = -S * ux * ux + 2 * ux * g, -S * uy * uy, -S * ux * uy + uy * g
        B1, B2 = 0.5 * (N[0] - N[2]), N[1]
        new = []
        for i in range(9):
            x, y = CX[i], CY[i]
            cu = x * ux + y * uy
            qy = x * x * Yxx + y * y * Yyy + 2 * x * y * Yxy - (Yxx + Yyy) / 3
            eq = req + rq * (3 * cu + 4.5 * cu * cu - 1.5 * (ux * ux + uy * uy))
            F = k2 * (S + 3 * x * g + 4.5 * qy) + self.k1 * ((x * x - y * y) * B1 + 2 * x * y * B2)
            new.append(n[i] + om * (W[i] * eq - n[i]) + W[i] * F)
        rho = 1 + req - drho
        vx, vy = jx / rho, jy / rho
        self.d, self.drho, self.phi = torch.stack(new), drho, phi
        if self.mode:
            self.sig = list(s)
        return torch.stack([vx.sum() / self.nx, torch.sqrt((vx * vx + vy * vy).max())])


def _network(x, w):
    """(hidden 1, hidden 2, output) with the working weights: the matrices and no biases in BF16."""
    (w1, b1), (w2, b2), (w3, b3) = w
    r = lambda t: t.float().to(torch.bfloat16).double()  # noqa: E731
    a1 = torch.tanh(x @ r(w1).T + b1)
    a2 = torch.tanh(a1 @ r(w2).T + b2)
    return a1, a2, a2 @ r(w3).T + b3


def _split(p):
    out, o = [], 0
    for n, i in ((H, N_IN), (H, H), (N_OUT, H)):
        out.append((p[o:o + n * i].reshape(n, i), p[o + n * i:o + n * i + n]))
        o += n * i + n
    return out


def _exact_train(case, seed):
    p = _weights(seed).double()
    x, y = (t.double() for t in _batches(case, seed))
    m, v, loss = torch.zeros_like(p), torch.zeros_like(p), None
    for k in range(case["steps"]):
        w = _split(p)
        a1, a2, out = _network(x[k], w)
        r = lambda t: t.float().to(torch.bfloat16).double()  # noqa: E731
        loss = ((out - y[k]) ** 2).mean()
        dy = 2 * (out - y[k]) / out.numel()
        d2 = (dy @ r(w[2][0])) * (1 - a2 * a2)
        d1 = (d2 @ r(w[1][0])) * (1 - a1 * a1)
        g = torch.cat([(d1.T @ x[k]).reshape(-1), d1.sum(0), (d2.T @ a1).reshape(-1), d2.sum(0),
                       (dy.T @ a2).reshape(-1), dy.sum(0)])
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        t = k + 1
        p = p - LR * (m / (1 - 0.9 ** t)) / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
    return {"params": p.numpy(), "loss": np.float64(loss)}


def _closed_form(p):
    """Steady profile of one channel on its rows: (u_x, N1), and on the network grid with its scales."""
    ny, hh = p["ny"], p["ny"] / 2.0
    w = p["g_x"] * hh / p["G_inf"]
    d = np.linspace(0.0, 1.0, 4001)
    b = p["gamma_c"] * (1 + p["theta"]) / (2 * p["theta"])
    dv = -w * d / 2 + b - np.sqrt((w * d / 2 - b) ** 2 + w * d * p["gamma_c"] / p["theta"])
    v = np.concatenate([[0.0], np.cumsum(0.5 * (dv[1:] + dv[:-1]) * np.diff(d))])
    v -= v[-1]
    dy = (np.arange(ny) - (ny - 1) / 2.0) / hh
    u = hh / p["tau0"] * np.interp(np.abs(dy), d, v)
    gd = np.interp(np.abs(dy), d, dv) / p["tau0"]
    tau = p["theta"] * p["tau0"]
    n1 = 2 * p["G_inf"] * (gd * tau / (1 + tau * np.abs(gd) / p["gamma_c"])) ** 2
    grid = (np.arange(GRID) + 0.5) / GRID * 2 - 1
    return dy, grid, [np.interp(grid, dy, f) for f in (u, n1)]


def _exact_warmstart(case, seed):
    ps = _sweep_params(case["channels"], case["ny_lo"], case["ny_hi"], seed)
    pred = _network(_features(ps).double(), _split(_weights(seed).double()))[2]
    mu, sd = (t.double() for t in _standardisation(seed))
    y = (pred * sd + mu).numpy()
    ux, dr = [], []
    for k, p in enumerate(ps):
        dy, grid, (u, n1) = _closed_form(p)
        pu = u + max(np.abs(u).max(), 1e-300) * y[k, :GRID]
        pn = n1 + max(np.abs(n1).max(), 1e-300) * y[k, 2 * GRID:]
        ux.append(np.interp(dy, grid, pu))
        dr.append(-1.5 * np.interp(dy, grid, pn))
    ex = _Exact(4, [p["ny"] for p in ps], ps)
    u = torch.from_numpy(np.concatenate(ux)).to(ex.dev)[:, None].expand(-1, 4) - 0.5 * ex.g  # j = rho u with its half force
    ex.drho = torch.from_numpy(np.concatenate(dr)).to(ex.dev)[:, None].expand(-1, 4).contiguous()
    ex.d = torch.stack([W[i] * (3 * CX[i] * u + (4.5 * CX[i] ** 2 - 1.5) * u * u) for i in range(9)])
    fu, _, fr = ex.fields()
    return {"pred": pred, "u": fu, "rho": fr}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "warmstart":
        return _exact_warmstart(case, seed)
    if kind == "sweep":
        ps = _sweep_params(case["channels"], case["ny_lo"], case["ny_hi"], seed)
        ex = _Exact(4, [p["ny"] for p in ps], ps)
        ex.d = torch.zeros(9, ex.rows, 4, dtype=torch.float64, device=ex.dev)
        for _ in range(case["steps"]):
            ex.step()
        u, sig, rho = ex.fields()
        return {"u": u, "sigma": sig, "rho": rho, "steps": None}
    p = _params(case, seed)
    if kind == "transient":
        ex = _Exact(case["nx"], [case["ny"]], [p])
        ex.start(p["seed"], AMP)
        mon = []
        for k in range(case["steps"]):
            ex.g = torch.tensor(_drive(p, k, case["steps"]), dtype=torch.float64, device=ex.dev)
            mon.append(ex.step())
        u, sig, rho = ex.fields()
        return {"u": u, "sigma": sig, "rho": rho, "flux_max": torch.stack(mon)}
    ex = _Exact(case["nx"], [case["ny"]], [p], case["x_mode"], case["walls"], case["stress_mode"],
                RELAX if case["relaxation"] else None, U_WALL)
    ex.start(p["seed"], AMP)
    for _ in range(case["steps"]):
        ex.step()
    u, sig, rho = ex.fields()
    return {"u": u, "sigma": sig, "rho": rho}
