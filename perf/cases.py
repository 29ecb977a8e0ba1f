"""The work that performance is measured on: forward runs and their log-likelihoods in both
precisions, a whole TMCMC stage, the surrogate's training step and log-likelihood, and a flow
field, each through the package's public entry points.

A case is a dict of plain values; ``listed()`` gives the fixed ones, ``draw(rng)`` another of
the same ranges, ``prepare(case, seed)`` what a user's program holds before the call,
``run(state)`` one pass, ``work(case)`` the bytes and operations a pass cannot do without, and
``exact(case, seed)`` the floating outputs in 64 bits from plain torch.

Forward Euler is stable only below a time step that falls with ds^3 / K_C, so every case takes
dt = 1e-4 / 2^p with the smallest p that keeps K_C = 10^0.2 stable, and priors that stay there:
a run on the edge of stability amplifies its own rounding, and its outputs say nothing.
Horizons are 2000 steps and less where a study takes 2e4 and more, so that a pass stays short.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1910_12007_gb300 as g
import synthetic
from paper_1910_12007_gb300 import surrogate as sg
from paper_1910_12007_gb300.api import MLP_HIDDEN, MLP_IN, MLP_OUT

STAGE_LO, STAGE_HI = (0.5, -0.3, 0.08), (5.0, 0.2, 0.12)   # posterior-like samples
PRIOR_LO, PRIOR_HI = (0.0, -1.0, 0.05), (10.0, 0.0, 0.2)   # the prior, where every run finishes
SWEEP_LO, SWEEP_HI = (0.0, -1.0, 0.05), (50.0, 0.0, 0.2)   # the sweep over the resistance
SPERM_LO, SPERM_HI = (0.0, 0.6, 0.08), (5.0, 0.95, 0.12)   # the full sperm model, K_C in [4, 9]
UNEVEN_N = (64, 128, 256, 512)
UNEVEN_DS = 1.0 / 255
SIGMA = 0.025  # 5 % of the head position's mean magnitude (L / 2)


# -------------------------------------------------------------------------------------
# cases
# -------------------------------------------------------------------------------------
def _forward(name, precision, n, batch, steps, obs_every, prior="stage", model="flagellum", output="loglik",
             uneven=False):
    c = {"kind": "forward", "precision": precision, "n": n, "batch": batch, "steps": steps, "obs_every": obs_every,
         "prior": prior, "model": model, "output": output, "uneven": uneven}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one forward run in FP64: the smallest call, a program looking at a single swimmer
        _forward("single_run_fp64", "fp64", 64, 1, 2000, 100, prior="prior", output="trajectory"),
        # a few dozen runs: the last chain steps of a TMCMC stage, a user's own small study
        _forward("few_runs_fp32", "fp32c", 128, 40, 2000, 50),
        # the log-likelihoods of one TMCMC batch (the headline workload's shape)
        _forward("stage_batch_fp32", "fp32c", 128, 1024, 2000, 50),
        # the same batch in FP64, the form that FP32 is judged by
        _forward("stage_batch_fp64", "fp64", 128, 1024, 200, 50),
        # samples of unequal length at a fixed ds in one launch
        _forward("uneven_batch_fp32", "fp32c", 512, 4096, 800, 100, prior="prior", uneven=True),
        # the sweep over the resistance with long flagella
        _forward("large_sweep_fp32", "fp32c", 1024, 256, 250, 50, prior="sweep", output="trajectory"),
        # the full sperm model (flagellum, head, neck), 2000 samples a stage, head velocities
        _forward("sperm_batch_fp32", "fp32c", 74, 2000, 2000, 100, prior="sperm", model="sperm"),
        # two sperm models coupled by the fluid, FP64, tail and head distances
        _forward("two_sperm_fp64", "fp64", 148, 152, 400, 50, prior="sperm", model="pair", output="trajectory"),
        # a whole TMCMC stage: analysis, resampling, the Metropolis chains' forward runs
        {"name": "tmcmc_stage_fp32", "kind": "stage", "n": 128, "batch": 1024, "steps": 2000, "obs_every": 50},
        # one step of the surrogate's training: forward, backward, Adam
        {"name": "surrogate_train", "kind": "train", "rows": 2048},
        # the surrogate's log-likelihood of a delayed-acceptance stage's proposals
        {"name": "surrogate_loglik", "kind": "surrogate", "batch": 4096},
        # velocity and pressure on a grid around one sperm model
        {"name": "flow_field", "kind": "flow", "nx": 512, "ny": 512, "points": 74},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _fit(fp64, n, batch, steps):
    """batch and steps cut until a pass stays below the largest listed one: the runs of a batch
    spread over the processors, about 150 at a time."""
    cap = 1.2e7 if fp64 else 4e8  # pair evaluations one after the other
    while n * n * steps * math.ceil(batch / 150) > cap:
        if batch > 150:
            batch = max(150, batch // 2)
        else:
            steps //= 2
    return batch, steps


def draw(rng):
    kind = rng.choice(("fp32", "fp32", "fp32", "fp64", "fp64", "uneven", "sperm", "stage", "train", "surrogate",
                       "flow"))
    if kind == "train":
        return {"kind": "train", "rows": _log_int(rng, 64, 4096)}
    if kind == "surrogate":
        return {"kind": "surrogate", "batch": _log_int(rng, 1, 8192)}
    if kind == "flow":
        return {"kind": "flow", "nx": _log_int(rng, 16, 512), "ny": _log_int(rng, 16, 512),
                "points": rng.randint(24, 150)}
    if kind == "stage":
        return {"kind": "stage", "n": rng.randint(32, 160), "batch": _log_int(rng, 128, 1024), "steps": 1000,
                "obs_every": 50}
    if kind == "sperm":
        fp64 = rng.random() < 0.3
        model = rng.choice(("sperm", "pair"))
        n = 74 if model == "sperm" else 148
        batch = _log_int(rng, 1, 1000 if fp64 else 2000)
        batch, steps = _fit(fp64, n, batch, rng.choice((100, 400) if fp64 else (400, 1500)))
        return _forward(None, "fp64" if fp64 else "fp32c", n, batch, steps, 50, "sperm", model,
                        rng.choice(("loglik", "trajectory")) if fp64 else "loglik")
    if kind == "uneven":
        return _forward(None, "fp32c", rng.choice((256, 512)), _log_int(rng, 64, 4096), rng.choice((200, 600)), 100, "prior",
                        uneven=True)
    n = min(1024, _log_int(rng, 24, 1024))
    if kind == "fp64":
        n = min(n, 300)
    prior = rng.choice(("stage", "prior", "sweep"))
    batch, steps = _fit(kind == "fp64", n, _log_int(rng, 1, 2000), rng.choice((200, 600, 1500)))
    return _forward(None, "fp64" if kind == "fp64" else "fp32c", n, batch, steps, 25, prior,
                    output="trajectory" if kind == "fp64" and rng.random() < 0.5 else "loglik")


# -------------------------------------------------------------------------------------
# what a program holds before the call
# -------------------------------------------------------------------------------------
def _time_step(ds):
    """dt = 1e-4 / 2^p: half the step at K_C = 1 that forward Euler allows, at spacing ds."""
    lam = 7.65e4 * max(1.0, (1.0 / 63 / ds) ** 3)
    return 1e-4 / 2 ** max(3, math.ceil(math.log2(1e-4 * lam)))


def _config(case):
    prec = g.FP64 if case.get("precision") == "fp64" else g.FP32C
    n, steps, every = case["n"], case["steps"], case["obs_every"]
    if case.get("model", "flagellum") != "flagellum":
        kw = dict(n_max=n, length=1.0, delta_over_ds=0.045 * 49, dt=1e-4 / 8, k_t=1e4, omega=4 * math.pi, n_head=24,
                  k_head_tens=1e4, k_head_c=0.8, k_neck_tens=500.0, k_neck_ang=1e4, obs_kind=g.OBS_HEAD_VELOCITY)
        if case["model"] == "pair":
            kw.update(obs_kind=g.OBS_PAIR_DISTANCES, n_swimmers=2, swimmer_distance=0.5, sigma_ratio=2.0)
    elif case.get("uneven"):
        kw = dict(n_max=n, ds_fixed=UNEVEN_DS, dt=_time_step(UNEVEN_DS))
    else:
        kw = dict(n_max=n, length=1.0, dt=_time_step(1.0 / (n - 1)))
    return g.SwimmerConfig(b_max=case["batch"], steps=steps, obs_every=every, precision=prec, **kw)


def _with_speed(case):
    """The mean speed is asked for where the swimmer moves far enough for it to mean something:
    over shorter horizons the displacement is near the positions' own rounding."""
    return case["precision"] == "fp64" and case["steps"] * _config(case).dt > 2e-3


def _box(prior):
    return {"stage": (STAGE_LO, STAGE_HI), "prior": (PRIOR_LO, PRIOR_HI), "sweep": (SWEEP_LO, SWEEP_HI),
            "sperm": (SPERM_LO, SPERM_HI)}[prior]


def _samples(case, seed):
    """theta [B, 3], points per sample [B] or None, and the observations with their noise (NumPy)."""
    theta = synthetic.prior_samples(seed, *_box(case.get("prior", "stage")), case["batch"])
    n_pts = None
    if case.get("uneven"):
        n_pts = synthetic.choice_n(seed, [k for k in UNEVEN_N if k <= case["n"]], case["batch"]).astype(np.int32)
    n_obs = case["steps"] // case["obs_every"]
    noise = synthetic.normals(seed, synthetic.NOISE, 0, 2 * n_obs).reshape(n_obs, 2)
    model = case.get("model", "flagellum")
    if model == "flagellum":
        # the head starts at (L, 0) and moves far less than the noise over these horizons
        mean, sigma = np.array([1.0, 0.0]), SIGMA
    elif model == "sperm":
        # head-centre velocities: the first moments' are of this size, 10 % noise
        mean, sigma = np.array([-5.0, 3.0]), 0.4
    else:
        mean, sigma = np.array([0.5, 0.5]), 0.05
    return theta, n_pts, mean + sigma * noise, sigma


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    put = lambda a, dt=torch.float64: torch.as_tensor(np.ascontiguousarray(a), device=dev).to(dt)
    kind = case["kind"]
    if kind == "forward":
        theta, n_pts, obs, sigma = _samples(case, seed)
        return {"kind": kind, "handle": g.swimmer_init(_config(case)), "theta": put(theta), "obs": put(obs),
                "sigma": sigma, "n_pts": None if n_pts is None else put(n_pts, torch.int32),
                "output": case["output"], "speed": _with_speed(case)}
    if kind == "stage":
        theta, _, obs, sigma = _samples(case, seed)
        h = g.swimmer_init(_config(case))
        s = {"kind": kind, "handle": h, "theta": put(theta), "obs": put(obs), "sigma": sigma}
        s["loglik"], _ = g.loglik_batch(h, s["theta"], s["obs"], sigma)
        u_res, u_acc, z = synthetic.stage_randoms(seed, 0, case["batch"], 3)
        s["uniforms"], s["normals"] = put(np.concatenate([u_res[None, :], u_acc])), put(z)
        return s
    if kind == "train":
        x, t, params, m, v = _train_inputs(case, seed)
        put32 = lambda a: put(a, torch.float32)
        return {"kind": kind, "x": put32(x), "t": put32(t), "params": put32(params), "m": put32(m), "v": put32(v),
                "workspace": g.mlp_workspace(case["rows"], dev),
                "grad": torch.empty(params.size, dtype=torch.float32, device=dev),
                "loss": torch.empty(1, dtype=torch.float32, device=dev)}
    if kind == "surrogate":
        theta, params, mean, std, obs = _surrogate_inputs(case, seed)
        h = g.swimmer_init(g.SwimmerConfig(n_max=128, b_max=case["batch"], dt=1e-4 / 64, steps=400, obs_every=10,
                                           precision=g.FP32C))
        g.swimmer_surrogate_set(h, put(params, torch.float32), *_surrogate_box(), mean, std, 1, 3.0, 2 * math.pi)
        return {"kind": kind, "handle": h, "theta": put(theta), "obs": put(obs)}
    state, grid, alpha = _flow_inputs(case, seed)
    h = g.swimmer_init(g.SwimmerConfig(n_max=74, b_max=1, steps=1, obs_every=1, precision=g.FP64))
    return {"kind": kind, "handle": h, "state": put(state), "grid": put(grid), "alpha": alpha}


def _train_inputs(case, seed):
    """Normalized inputs and targets of one batch, the weights and Adam's moments in mid-training."""
    n = case["rows"]
    x = 2.0 * synthetic.uniforms(seed, synthetic.TRAIN, 0, n * MLP_IN).reshape(n, MLP_IN) - 1.0
    x[:, 3:] = 0.0  # tension stiffness and frequency are fixed in a training set
    t = synthetic.normals(seed, synthetic.TRAIN, 1, n * MLP_OUT).reshape(n, MLP_OUT)
    params = sg.init_params(seed % 65536, "cpu").numpy()
    m = 1e-4 * synthetic.normals(seed, synthetic.TRAIN, 2, params.size)
    v = 1e-7 * (0.5 + synthetic.uniforms(seed, synthetic.TRAIN, 3, params.size))
    return tuple(np.asarray(a, dtype=np.float32) for a in (x, t, params, m, v))


def _surrogate_box():
    lo = [*PRIOR_LO, 3.0, 2 * math.pi]
    return lo, [10.0, 1.0, 0.2, 3.0, 2 * math.pi]


def _surrogate_inputs(case, seed):
    theta = synthetic.prior_samples(seed, STAGE_LO, STAGE_HI, case["batch"])
    params = sg.init_params(seed % 65536, "cpu").numpy()
    # trajectories stay near the head's start, with the spread of a short horizon
    mean = np.tile([1.0, 0.0], MLP_OUT // 2) + 1e-3 * synthetic.normals(seed, synthetic.NOISE, 1, MLP_OUT)
    std = 1e-3 * (0.5 + synthetic.uniforms(seed, synthetic.NOISE, 2, MLP_OUT))
    obs = np.array([1.0, 0.0]) + SIGMA * synthetic.normals(seed, synthetic.NOISE, 3, MLP_OUT).reshape(-1, 2)
    return theta, params, mean, std, obs


def _flow_inputs(case, seed):
    """A bent swimmer of `points` points with balanced forces, and the grid around it."""
    n = case["points"]
    u = synthetic.uniforms(seed, synthetic.PRIOR, 3, 3)
    s = np.linspace(0.0, 1.0 + 0.3 * u[0], n)
    y = 0.1 * (1.0 - 0.5 * s) * np.sin(2 * math.pi * (s - u[1]))
    f = synthetic.normals(seed, synthetic.PRIOR, 4, 2 * n).reshape(n, 2)
    f -= f.mean(0)
    xs, ys = np.linspace(-0.5, 2.0, case["nx"]), np.linspace(-1.25, 1.25, case["ny"])
    grid = np.stack(np.meshgrid(xs, ys, indexing="ij"), axis=-1).reshape(-1, 2)
    return np.stack([s, y, f[:, 0], f[:, 1]], axis=1), grid, 0.2 + 4.0 * float(u[2])


FLOW_DELTA, FLOW_REACH = 0.045, 4.0
LEARNING_RATE, ADAM_STEP = 2e-3, 100


# -------------------------------------------------------------------------------------
# one pass
# -------------------------------------------------------------------------------------
def run(s):
    kind = s["kind"]
    if kind == "forward":
        if s["output"] == "loglik":
            return g.loglik_batch(s["handle"], s["theta"], s["obs"], s["sigma"], n_pts=s["n_pts"])
        if s["speed"]:
            return g.forward_batch(s["handle"], s["theta"], s["n_pts"])
        # trajectories and status alone, as a training set keeps them
        B, dev = s["theta"].shape[0], s["theta"].device
        out = (torch.empty((B, s["handle"].cfg.n_obs, 2), dtype=torch.float64, device=dev), None,
               torch.empty(B, dtype=torch.int32, device=dev))
        return g.forward_batch(s["handle"], s["theta"], s["n_pts"], out=out)
    if kind == "stage":
        st = g.TmcmcState(s["theta"].clone(), s["loglik"].clone(), s["obs"], s["sigma"], STAGE_LO, STAGE_HI)
        r = g.tmcmc_stage(s["handle"], st, s["uniforms"], s["normals"])
        return [st.theta, st.loglik, st.status, r["q"], r["log_s"], torch.tensor(r["mu"], dtype=torch.float64),
                r["unique"], r["n_accept"], r["n_exact_path"]]
    if kind == "train":
        g.mlp_backward(s["params"], s["x"], s["t"], workspace=s["workspace"], grad=s["grad"], loss=s["loss"])
        g.mlp_adam(s["params"], s["grad"], s["m"], s["v"], ADAM_STEP, LEARNING_RATE)
        return [s["grad"], s["loss"], s["params"], s["m"], s["v"]]
    if kind == "surrogate":
        return g.surrogate_loglik_batch(s["handle"], s["theta"], s["obs"], SIGMA)
    return g.swimmer_flow_field(s["handle"], s["alpha"], FLOW_DELTA, FLOW_REACH, s["state"], s["grid"])


# -------------------------------------------------------------------------------------
# what a pass cannot do without
# -------------------------------------------------------------------------------------
# one unordered pair: separation 2, u 4, two kernel functions 8, the symmetric 2 x 2 mobility 7,
# 8 per direction; forces and the position update of a point, about 200
PAIR_FLOPS, POINT_FLOPS = 37, 200
MLP_MACS = 5 * 256 + 2 * 256 * 256 + 256 * 80


def work(case):
    kind = case["kind"]
    if kind in ("forward", "stage"):
        n, B = float(case["n"]), case["batch"]
        n2 = n * n
        if case.get("uneven"):
            some = [k for k in UNEVEN_N if k <= case["n"]]
            n, n2 = sum(some) / len(some), sum(k * k for k in some) / len(some)
        n_obs = case["steps"] // case["obs_every"]
        out = 12.0 if case.get("output", "loglik") == "loglik" else 16.0 * n_obs + 4
        flops = B * case["steps"] * (PAIR_FLOPS * (n2 - n) / 2 + POINT_FLOPS * n)
        if kind == "stage":  # theta, log-likelihood, uniforms and normals in, both and the status out
            return {"bytes": B * (32.0 + 24 + 24 + 36) + 16.0 * n_obs, "flops": flops}
        return {"bytes": B * (24.0 + out + (4 if case.get("uneven") else 0)) + 16.0 * n_obs, "flops": flops}
    if kind == "train":
        n, p = case["rows"], g.MLP_NPARAM
        return {"bytes": 4.0 * (n * (MLP_IN + MLP_OUT) + 7 * p), "flops": 6.0 * n * MLP_MACS}
    if kind == "surrogate":
        return {"bytes": case["batch"] * 32.0 + 4.0 * g.MLP_NPARAM, "flops": 2.0 * case["batch"] * MLP_MACS}
    G = case["nx"] * case["ny"]
    return {"bytes": 40.0 * G + 32.0 * case["points"], "flops": 50.0 * G * case["points"]}


# -------------------------------------------------------------------------------------
# the same outputs in 64 bits, plain torch
# -------------------------------------------------------------------------------------
EXACT_PAIRS = 7e10  # ordered pair evaluations that stay inside 20 seconds


def exact(case, seed):
    kind = case["kind"]
    if kind == "forward":
        return _exact_forward(case, seed)
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "surrogate":
        return _exact_surrogate(case, seed)
    if kind == "flow":
        return _exact_flow(case, seed)
    return None  # a stage: hundreds of forward runs one after the other


class _Kernel:
    """g1 = B'' and g2 = (r B'' - B') / r^3 of the regularized Brinkmanlet for a batch of
    (alpha, delta), as piecewise polynomials in u = 1 + r^2 / delta^2 fitted to the solution of
    the radial problem by variation of parameters (16-point Gauss-Legendre integrals between
    Chebyshev nodes), 8 pieces an octave."""

    SUB, N = 8, 12

    def __init__(self, alpha, delta, reach):
        B, dev = alpha.numel(), alpha.device
        f64 = dict(dtype=torch.float64, device=dev)
        self.delta = delta
        octaves = int(torch.floor(torch.log2(1.0 + (reach / delta).square().max())).item()) + 1
        self.panels = octaves * self.SUB
        k = np.arange(self.N)
        t = np.cos(math.pi * (k[::-1] + 0.5) / self.N)  # ascending nodes
        p = np.arange(self.panels)
        lo = 2.0 ** (p // self.SUB) * (1.0 + (p % self.SUB) / self.SUB)
        u = lo[:, None] + 2.0 ** (p // self.SUB)[:, None] / self.SUB * 0.5 * (t[None, :] + 1.0)
        u = torch.tensor(u.reshape(1, -1), **f64)
        d, a = delta[:, None], alpha[:, None]
        r = d * torch.sqrt(u - 1.0)
        gx, gw = (torch.tensor(v, **f64) for v in np.polynomial.legendre.leggauss(16))
        phi_s = lambda s, dd: s * 3.0 * dd ** 3 / (2.0 * math.pi * (s * s + dd * dd) ** 2.5)

        def integrals(f, lo_, hi_):
            half = 0.5 * (hi_ - lo_)[..., None]
            s = 0.5 * (hi_ + lo_)[..., None] + half * gx
            return (f(a[..., None] * s) * phi_s(s, d[..., None]) * half * gw).sum(-1)

        A = torch.cumsum(integrals(_i0m1, torch.cat([torch.zeros_like(r[:, :1]), r[:, :-1]], 1), r), 1)
        C = integrals(torch.special.modified_bessel_k0, r[:, :-1], r[:, 1:])
        end = torch.log1p(60.0 / (a * r[:, -1:]))
        edge = r[:, -1:] * torch.exp(end * torch.linspace(0, 1, 97, **f64))
        tail = integrals(torch.special.modified_bessel_k0, edge[:, :-1], edge[:, 1:]).sum(1, keepdim=True)
        C = torch.flip(torch.cumsum(torch.flip(torch.cat([C, tail], 1), [1]), 1), [1])
        x = a * r
        k0, k1 = torch.special.modified_bessel_k0(x), torch.special.modified_bessel_k1(x)
        i0 = torch.special.i0(x)
        i2 = _i2(x)
        k2 = k0 + 2.0 * k1 / x
        t2k2 = torch.where(x <= 2.0, _two_over_x2_less_k2(x.clamp(max=2.0)), 2.0 / (x * x) - k2)
        R = torch.sqrt(r * r + d * d)
        M0 = (r * r / (R + d)) * (R * R + R * d + d * d) / R ** 3 / (2.0 * math.pi)
        g1 = 0.5 * (t2k2 - k0) * M0 - 0.5 * (k0 + k2) * A - 0.5 * (i0 + i2) * C
        g2 = (t2k2 * M0 - k2 * A - i2 * C) / (r * r)
        # Chebyshev coefficients on each piece, then powers of its local coordinate in [-1, 1]
        T = np.polynomial.chebyshev.chebvander(t, self.N - 1)
        w = np.full(self.N, 2.0 / self.N)
        w[0] = 1.0 / self.N
        powers = np.zeros((self.N, self.N))
        for i in range(self.N):
            c = np.polynomial.chebyshev.cheb2poly(np.eye(self.N)[i])
            powers[i, :c.size] = c
        to_cheb, to_poly = torch.tensor(T * w, **f64), torch.tensor(powers, **f64)
        fit = lambda v: ((v.reshape(B, self.panels, self.N) @ to_cheb) @ to_poly).reshape(B * self.panels, self.N)
        self.c1, self.c2 = (fit(v).T.contiguous() for v in (g1, g2))

    def __call__(self, r2, rows):
        """g1, g2 at squared distances r2 [b, ...] of the samples `rows` (a slice)."""
        shape = (-1,) + (1,) * (r2.dim() - 1)
        u = 1.0 + r2 / (self.delta[rows] ** 2).reshape(shape)
        bits = u.view(torch.int64)
        panel = ((bits >> 49) - (1023 << 3)).clamp_(max=self.panels - 1)
        local = ((bits << 3) & 0x000FFFFFFFFFFFFF) | 0x3FF0000000000000
        t = local.view(torch.float64) * 2.0 - 3.0
        base = torch.arange(rows.start, rows.stop, device=r2.device).reshape(shape) * self.panels
        at = (panel + base).reshape(-1)
        out = []
        for c in (self.c1, self.c2):
            v = c[-1].take(at)
            for k in range(self.N - 2, -1, -1):
                v = torch.addcmul(c[k].take(at), v, t.reshape(-1))
            out.append(v.reshape(r2.shape))
        return out


def _i0m1(x):
    y = 0.25 * x.clamp(max=1.5) ** 2
    term, s = y, torch.zeros_like(y)
    for k in range(1, 20):
        s = s + term
        term = term * y / (k + 1.0) ** 2
    return torch.where(x < 1.5, s, torch.special.i0(x) - 1.0)


def _i2(x):
    y = 0.25 * x.clamp(max=4.0) ** 2
    term, s = 0.5 * y, torch.zeros_like(y)
    for k in range(40):
        s = s + term
        term = term * y / ((k + 1.0) * (k + 3.0))
    return torch.where(x < 4.0, s, torch.special.i0(x) - 2.0 * torch.special.i1(x) / x)


def _two_over_x2_less_k2(x):
    """2/x^2 - K2(x) for x <= 2 from the ascending series of K2 (no cancellation)."""
    y = 0.25 * x * x
    harmonic = lambda m: sum(1.0 / j for j in range(1, m + 1))
    term, s = 0.5 * torch.ones_like(y), torch.zeros_like(y)
    for k in range(24):
        s = s + (harmonic(k) + harmonic(k + 2) - 2.0 * 0.57721566490153286061) * term
        term = term * y / ((k + 1.0) * (k + 3.0))
    return 0.5 + torch.log(0.5 * x) * _i2(x) - 0.5 * y * s


class _Swimmers:
    """Forward runs of one size: initial points, elastic energy, observations."""

    def __init__(self, cfg, nf, theta):
        dev = theta.device
        self.cfg, self.nf, self.nh = cfg, nf, cfg.n_head
        self.length = (nf - 1) * cfg.ds_fixed if cfg.ds_fixed > 0 else cfg.length
        self.ds = self.length / (nf - 1)
        self.delta = cfg.delta_over_ds * self.ds
        self.alpha, self.kc, self.amp = theta[:, 0], 10.0 ** theta[:, 1:2], theta[:, 2:3]
        x = torch.arange(nf, dtype=torch.float64, device=dev) * self.ds
        X = torch.stack([x, torch.zeros_like(x)], 1)
        reach = self.length
        if self.nh:
            self.hr = self.nh * self.ds / (2.0 * math.pi)
            th = 2.0 * math.pi * torch.arange(self.nh, dtype=torch.float64, device=dev) / self.nh
            head = torch.stack([self.length + self.ds + self.hr + self.hr * torch.cos(th), self.hr * torch.sin(th)], 1)
            X = torch.cat([X, head])
            reach += self.ds + 2.0 * self.hr
            h2 = self.nh // 2
            H = lambda m: nf + m % self.nh
            pairs = [(H(m), H(m + 1), cfg.k_head_tens) for m in range(self.nh)]
            pairs += [(H(m), H(m + h2), cfg.k_head_tens) for m in range(h2)]
            pairs += [(nf - 1, H(h2 + q), cfg.k_neck_tens) for q in (-1, 0, 1)]
            pairs += [(nf - 2, H(h2 + q), cfg.k_neck_tens) for q in (-1, 1)]
            self.si, self.sj = (torch.tensor([p[q] for p in pairs], device=dev) for q in (0, 1))
            self.sk = torch.tensor([p[2] for p in pairs], dtype=torch.float64, device=dev)
            self.sl = (X[self.sj] - X[self.si]).norm(dim=1)
        self.per = X.shape[0]
        if cfg.n_swimmers == 2:
            X = torch.cat([X, X + torch.tensor([0.0, cfg.swimmer_distance], dtype=torch.float64, device=dev)])
            reach += cfg.swimmer_distance
        self.reach = 1.25 * reach
        self.X0 = X
        self.s = x[1:-1]

    @staticmethod
    def _curvature(back, here, ahead, h):
        d1, d2 = (ahead - back) / (2.0 * h), (ahead - 2.0 * here + back) / (h * h)
        return (d1[..., 0] * d2[..., 1] - d1[..., 1] * d2[..., 0]) / d1.square().sum(-1) ** 1.5

    def energy(self, X, t):
        c, e = self.cfg, 0.0
        for k in range(c.n_swimmers):
            P = X[:, k * self.per:(k + 1) * self.per]
            F = P[:, :self.nf]
            e = e + c.k_t * self.ds * (((F[:, 1:] - F[:, :-1]).norm(dim=2) / self.ds - 1.0) ** 2).sum()
            ph = c.eta * self.s - c.omega * t
            want = -self.amp * (2.0 * c.eta / self.length * torch.cos(ph)
                                + (1.0 - self.s / self.length) * c.eta ** 2 * torch.sin(ph))
            zeta = self._curvature(F[:, :-2], F[:, 1:-1], F[:, 2:], self.ds)
            e = e + (self.kc * self.ds * (zeta - want) ** 2).sum()
            if self.nh:
                ell = (P[:, self.sj] - P[:, self.si]).norm(dim=2)
                e = e + (self.sk * self.sl * (ell / self.sl - 1.0) ** 2).sum()
                H = P[:, self.nf:]
                kap = self._curvature(H.roll(1, 1), H, H.roll(-1, 1), 2.0 * math.pi * self.hr / self.nh)
                e = e + c.k_head_c * (2.0 * math.pi * self.hr / self.nh) * ((kap - 1.0 / self.hr) ** 2).sum()
                h2 = self.nh // 2
                z = ((H[:, h2] - F[:, -1]) * (H[:, h2 + 1] - H[:, h2 - 1])).sum(1)
                e = e + c.k_neck_ang * (z * z).sum()
        return e

    def run(self):
        """Observations [B, n_obs, 2] and mean speed [B]."""
        c, B, n = self.cfg, self.alpha.numel(), self.X0.shape[0]
        dev = self.X0.device
        full = lambda v: torch.full((B,), v, dtype=torch.float64, device=dev)
        kern = _Kernel(self.alpha, full(self.delta), full(self.reach))
        X = self.X0.expand(B, n, 2).clone()
        chunk = max(1, int(2e7 // (n * n)))
        centre = lambda k: X[:, k * self.per + self.nf:(k + 1) * self.per].mean(1)
        at = lambda: centre(0) if self.nh else X[:, :self.nf].mean(1)
        start = at()
        last, obs = start, []
        for step in range(c.steps):
            Y = X.detach().requires_grad_(True)
            F = -torch.autograd.grad(self.energy(Y, step * c.dt), Y)[0]
            V = torch.empty_like(X)
            for b in range(0, B, chunk):
                rows = slice(b, min(B, b + chunk))
                d = X[rows, :, None, :] - X[rows, None, :, :]
                dx, dy = d[..., 0], d[..., 1]
                g1, g2 = kern(dx * dx + dy * dy, rows)
                fx, fy = F[rows, None, :, 0], F[rows, None, :, 1]
                w = (fx * dx + fy * dy) * g2
                V[rows, :, 0] = (w * dx - fx * g1).sum(2)
                V[rows, :, 1] = (w * dy - fy * g1).sum(2)
            X = X + (c.dt / c.mu) * V
            if (step + 1) % c.obs_every == 0:
                if c.obs_kind == g.OBS_HEAD_POINT:
                    obs.append(X[:, self.nf - 1].clone())
                elif c.obs_kind == g.OBS_HEAD_VELOCITY:
                    obs.append((at() - last) / (c.obs_every * c.dt))
                    last = at()
                else:
                    obs.append(torch.stack([(X[:, self.per] - X[:, 0]).norm(dim=1),
                                            (centre(1) - centre(0)).norm(dim=1)], 1))
        return torch.stack(obs, 1), (at() - start)[:, 0] / (c.steps * c.dt)


def _exact_forward(case, seed):
    theta, n_pts, obs, sigma = _samples(case, seed)
    cfg = _config(case)
    sizes = np.full(case["batch"], case["n"]) if n_pts is None else n_pts
    if float((sizes.astype(np.float64) ** 2).sum()) * case["steps"] > EXACT_PAIRS:
        return None
    dev = torch.device("cuda", torch.cuda.current_device())
    theta, obs = torch.tensor(theta, device=dev), torch.tensor(obs, device=dev)
    traj = torch.empty((case["batch"], cfg.n_obs, 2), dtype=torch.float64, device=dev)
    speed = torch.empty(case["batch"], dtype=torch.float64, device=dev)
    for n in sorted(set(sizes.tolist())):
        at = torch.tensor(np.flatnonzero(sizes == n), device=dev)
        nf = n // cfg.n_swimmers - cfg.n_head
        traj[at], speed[at] = _Swimmers(cfg, nf, theta[at]).run()
    if case["output"] == "trajectory":
        return traj, speed if _with_speed(case) else None, None
    ratio = cfg.sigma_ratio or 1.0
    res = (obs - traj) / torch.tensor([1.0, ratio], dtype=torch.float64, device=dev)
    J = res.square().sum((1, 2))
    return -cfg.n_obs * (math.log(2.0 * math.pi * sigma ** 2) + math.log(ratio)) - 0.5 * J / sigma ** 2, None


def _layers(flat):
    out, o = [], 0
    sizes = (MLP_IN, MLP_HIDDEN, MLP_HIDDEN, MLP_HIDDEN, MLP_OUT)
    for fi, fo in zip(sizes[:-1], sizes[1:]):
        out.append((flat[o:o + fo * fi].reshape(fo, fi), flat[o + fo * fi:o + fo * fi + fo]))
        o += fo * fi + fo
    return out


def _network(flat, x):
    layers = _layers(flat)
    for W, b in layers[:-1]:
        x = torch.nn.functional.gelu(x @ W.T + b)
    return x @ layers[-1][0].T + layers[-1][1]


def _exact_train(case, seed):
    x, t, params, m, v = (torch.tensor(a, dtype=torch.float64) for a in _train_inputs(case, seed))
    params.requires_grad_(True)
    loss = (_network(params, x) - t).square().mean()
    grad = torch.autograd.grad(loss, params)[0]
    m = 0.9 * m + 0.1 * grad
    v = 0.999 * v + 0.001 * grad * grad
    step = (m / (1 - 0.9 ** ADAM_STEP)) / (torch.sqrt(v / (1 - 0.999 ** ADAM_STEP)) + 1e-8)
    return [grad, loss.detach().reshape(1), params.detach() - LEARNING_RATE * step, m, v]


def _exact_surrogate(case, seed):
    theta, params, mean, std, obs = _surrogate_inputs(case, seed)
    lo, hi = (np.array(v) for v in _surrogate_box())
    x = np.zeros((case["batch"], MLP_IN))
    x[:, :3] = 2.0 * (theta - lo[:3]) / (hi - lo)[:3] - 1.0
    y = mean + std * _network(torch.tensor(params, dtype=torch.float64), torch.tensor(x)).numpy()
    J = ((obs.reshape(-1) - y) ** 2).sum(1)
    n_obs = MLP_OUT // 2
    return torch.tensor(-n_obs * math.log(2.0 * math.pi * SIGMA ** 2) - 0.5 * J / SIGMA ** 2)


def _exact_flow(case, seed):
    state, grid, alpha = _flow_inputs(case, seed)
    dev = torch.device("cuda", torch.cuda.current_device())
    state, grid = torch.tensor(state, device=dev), torch.tensor(grid, device=dev)
    one = lambda v: torch.tensor([v], dtype=torch.float64, device=dev)
    kern = _Kernel(one(alpha), one(FLOW_DELTA), one(FLOW_REACH))
    vel = torch.zeros_like(grid)
    pres = torch.zeros(grid.shape[0], dtype=torch.float64, device=dev)
    for q in state:
        d = grid - q[:2]
        r2 = d.square().sum(1)
        g1, g2 = (v[0] for v in kern(r2[None], slice(0, 1)))
        fd = d @ q[2:]
        vel += (fd * g2)[:, None] * d - g1[:, None] * q[2:]
        R = torch.sqrt(r2 + FLOW_DELTA ** 2)
        pres += fd * (R * R + R * FLOW_DELTA + FLOW_DELTA ** 2) / (2.0 * math.pi * R ** 3 * (R + FLOW_DELTA))
    return vel, pres
