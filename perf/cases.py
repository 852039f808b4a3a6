"""What the speed of this package is measured on: one pass of a user's call per case.

The systems are synthetic radial-velocity fits of the package's own workload
shapes (see ``paper_0812_2976_gb300/synth.py``): truths with log-uniform
periods and amplitudes, models scattered around them, one star's observations
for a uniform batch or each system's own for a ragged one.  Everything is
drawn on the GPU from the seed; no part of the package takes part in making
inputs or in ``exact``.

The differential-evolution MCMC step is not among the cases: its accept /
reject decisions are whole numbers that hang on the last bit of chi2, so two
correct builds may return different chains.  Its time is the chi2 call's.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_0812_2976_gb300 as kc

EPOCH = 2450000.0
TWO_PI = 2.0 * math.pi
MAX_PLANETS_RAGGED = 6
CHUNK = 1 << 24             # elements per step of the 64-bit evaluation


def listed():
    return [
        # A plain double-precision fit of one planet: the smallest call a user
        # makes; launches, latency and the call itself are all of its time.
        dict(name="chi2_fp64_small", kind="chi2", mode="fp64", n_sys=64, n_pl=1, n_obs=32,
             perturb=0.01, e_max=0.8, t0=0.0, jitter=0.0),
        # One ensemble of walkers of a sampler, odd sizes, with an epoch and a
        # fixed jitter: called over and over, far too small to fill the GPU.
        dict(name="chi2_mixed_ensemble", kind="chi2", mode="mixed", n_sys=300, n_pl=3, n_obs=101,
             perturb=0.01, e_max=0.8, t0=EPOCH, jitter=1.5),
        # The paper's batch, the headline of the benchmark: 4096 four-planet
        # models against 256 observations, absolute times (t0 = 0).
        dict(name="chi2_mixed_paper", kind="chi2", mode="mixed", n_sys=4096, n_pl=4, n_obs=256,
             perturb=0.01, e_max=0.8, t0=0.0, jitter=0.0),
        # A large grid search over wide perturbations and eccentricities.
        dict(name="chi2_mixed_sweep", kind="chi2", mode="mixed", n_sys=1 << 20, n_pl=4, n_obs=256,
             perturb=0.1, e_max=0.95, t0=0.0, jitter=0.0),
        # The paper's batch in double precision (final values, checks of the
        # mixed path).
        dict(name="chi2_fp64_paper", kind="chi2", mode="fp64", n_sys=4096, n_pl=4, n_obs=256,
             perturb=0.01, e_max=0.8, t0=0.0, jitter=0.0),
        # chi2 and its gradient for a large population of optimisers.
        dict(name="grad_mixed", kind="grad", mode="mixed", n_sys=65536, n_pl=3, n_obs=512,
             perturb=0.01, e_max=0.8, t0=EPOCH, jitter=0.0),
        # Double-precision refinement through autograd, odd sizes.
        dict(name="grad_fp64_autograd", kind="chi2_backward", mode="fp64", n_sys=1000, n_pl=5,
             n_obs=333, perturb=0.01, e_max=0.8, t0=EPOCH, jitter=0.0),
        # The normal equations of a Levenberg-Marquardt step.
        dict(name="gauss_newton_mixed", kind="gn", mode="mixed", n_sys=65536, n_pl=3, n_obs=512,
             perturb=0.01, e_max=0.8, t0=EPOCH, jitter=0.0),
        # The free-jitter likelihood and its gradient through autograd, the
        # target of a gradient-based sampler.
        dict(name="nll_mixed_autograd", kind="nll_backward", mode="mixed", n_sys=10000, n_pl=2,
             n_obs=150, perturb=0.01, e_max=0.8, t0=EPOCH, jitter=0.0),
        # A survey: every system its own star, planet count and observations.
        dict(name="ragged_grad_mixed", kind="ragged", mode="mixed", n_sys=50000, grad=True,
             obs_min=16, obs_max=1024, perturb=0.01, e_max=0.8),
        # Posterior-predictive velocity curves of 512 draws on a fine grid.
        dict(name="rv_predict", kind="predict", mode="fp64", n_sys=512, n_pl=3, n_obs=1000,
             perturb=0.01, e_max=0.8, t0=EPOCH),
        # Kepler's equation alone for arrays of (M, e): bound by memory.
        dict(name="kepler_mixed", kind="kepler", mode="mixed", n=1 << 24, e_max=0.95),
    ]


# (kind, mode): planet-observation evaluations a drawn case may have, so that
# none costs more than the largest listed one.
_DRAWN = {
    ("chi2", "mixed"): 5.0e8, ("chi2", "fp64"): 2.0e7, ("grad", "mixed"): 2.0e8,
    ("grad", "fp64"): 1.0e7, ("chi2_backward", "mixed"): 1.0e8, ("nll_backward", "mixed"): 1.0e8,
    ("gn", "mixed"): 1.0e8, ("ragged", "mixed"): 1.0e8, ("predict", "fp64"): 2.0e6,
    ("kepler", "mixed"): 6.0e7, ("kepler", "fp64"): 1.6e7,
}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind, mode = rng.choice(sorted(_DRAWN))
    cap = _DRAWN[kind, mode]
    e_max = rng.choice([0.3, 0.8, 0.95])
    if kind == "kepler":
        return dict(kind=kind, mode=mode, n=_log_int(rng, 1000, cap), e_max=e_max)
    perturb = rng.choice([0.001, 0.01, 0.1])
    if kind == "ragged":
        obs_min = _log_int(rng, 4, 64)
        obs_max = _log_int(rng, 2 * obs_min, 1024)
        most = cap / (0.5 * (obs_min + obs_max) * 3.5)
        return dict(kind=kind, mode=mode, n_sys=_log_int(rng, 200, min(50000, most)),
                    grad=rng.random() < 0.5, obs_min=obs_min, obs_max=obs_max, perturb=perturb,
                    e_max=e_max)
    n_pl = rng.randint(1, 8)
    n_obs = _log_int(rng, 16, 1024)
    case = dict(kind=kind, mode=mode, n_sys=_log_int(rng, 64, min(1 << 20, cap / (n_pl * n_obs))),
                n_pl=n_pl, n_obs=n_obs, perturb=perturb, e_max=e_max,
                t0=rng.choice([0.0, EPOCH]) if kind in ("chi2", "predict") else EPOCH)
    if kind in ("chi2", "grad", "chi2_backward", "gn", "nll_backward"):
        case["jitter"] = 0.0 if kind == "nll_backward" else rng.choice([0.0, 2.0])
    return case


# ------------------------------------------------------------ inputs

def _uniform(gen, shape, lo, hi):
    return lo + (hi - lo) * torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)


def _normal(gen, shape):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)


def _planets(gen, n, n_pl, e_max):
    """[n, n_pl, 5] truths (P, K, e, omega, M0)."""
    x = torch.empty((n, n_pl, 5), dtype=torch.float64, device="cuda")
    x[..., 0] = torch.exp(_uniform(gen, (n, n_pl), 0.0, math.log(4000.0)))
    x[..., 1] = torch.exp(_uniform(gen, (n, n_pl), 0.0, math.log(100.0)))
    x[..., 2] = _uniform(gen, (n, n_pl), 0.0, e_max)
    x[..., 3] = _uniform(gen, (n, n_pl), 0.0, TWO_PI)
    x[..., 4] = _uniform(gen, (n, n_pl), 0.0, TWO_PI)
    return x


def _scatter(gen, rows, n_pl, rel):
    """Model rows: every parameter of the truth scattered by ``rel``."""
    m = rows * (1.0 + rel * _normal(gen, rows.shape))
    end = 5 * n_pl
    m[:, 0:end:5].clamp_(min=1e-3)
    m[:, 1:end:5].clamp_(min=0.0)
    m[:, 2:end:5].clamp_(0.0, 0.95)
    return m


def _eccentric(M, e):
    """E - e sin E = M in 64 bits: Danby's quartic steps from his start."""
    M = M - TWO_PI * torch.round(M / TWO_PI)
    E = M + 0.85 * e * torch.where(M < 0, -1.0, 1.0)
    for _ in range(5):
        s, c = torch.sin(E), torch.cos(E)
        f, f1, f2, f3 = (E - M) - e * s, 1.0 - e * c, e * s, e * c
        d = -f / f1
        d = -f / (f1 + 0.5 * d * f2)
        d = -f / (f1 + 0.5 * d * f2 + d * d * f3 / 6.0)
        E = E + d
    return E


def _orbit(P, e, M0, dt):
    """sin E, cos E at the times dt after the epoch; fmod is exact, so the
    phase keeps its bits over millions of periods."""
    E = _eccentric(TWO_PI * (torch.fmod(dt, P) / P) + M0, e)
    return torch.sin(E), torch.cos(E)


def _velocity(P, K, e, w, M0, dt):
    s, c = _orbit(P, e, M0, dt)
    b2 = (1.0 - e) * (1.0 + e)
    return K * (b2 * torch.cos(w) * c - torch.sqrt(b2) * torch.sin(w) * s) / (1.0 - e * c)


def _partials(P, K, e, w, M0, dt):
    """The velocity and its derivatives by (P, K, e, omega, M0)."""
    s, c = _orbit(P, e, M0, dt)
    D = 1.0 - e * c
    b = torch.sqrt((1.0 - e) * (1.0 + e))
    cf, sf, cw, sw = (c - e) / D, b * s / D, torch.cos(w), torch.sin(w)
    cwf, swf = cw * cf - sw * sf, sw * cf + cw * sf
    dK = cwf + e * cw
    dM = -K * swf * b / (D * D)
    de = K * cw - K * swf * (s / D) * (1.0 / b + b / D)
    return K * dK, (dM * (-TWO_PI * dt / (P * P)), dK, de, -K * (swf + e * sw), dM)


def _uniform_inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n_pl, n_obs, t0 = case["n_pl"], case["n_obs"], case["t0"]
    t = torch.sort(_uniform(gen, (n_obs,), EPOCH, EPOCH + 4000.0)).values
    sigma = _uniform(gen, (n_obs,), 1.0, 5.0)
    truth = _planets(gen, 1, n_pl, case["e_max"])[0]
    truth[:, 0] = torch.sort(truth[:, 0]).values
    truth = truth.reshape(-1)
    gamma = _uniform(gen, (1,), -10.0, 10.0)
    row = torch.cat([truth, gamma])
    v = gamma + sigma * _normal(gen, (n_obs,))
    for j in range(n_pl):
        v = v + _velocity(*truth[5 * j:5 * j + 5], t - t0)
    params = _scatter(gen, row[None, :].expand(case["n_sys"], -1), n_pl, case["perturb"])
    if case["kind"] == "nll_backward":
        params = torch.cat([params, _uniform(gen, (case["n_sys"], 1), 0.5, 3.0)], dim=1)
    return params.contiguous(), t, v, sigma


def _ragged_inputs(case, seed):
    # the sizes belong to the case (the outputs' shapes follow from them), the
    # values to the seed
    host = np.random.default_rng([case["n_sys"], case["obs_min"], case["obs_max"]])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n, top = case["n_sys"], MAX_PLANETS_RAGGED
    n_pl = host.integers(1, top + 1, n).astype(np.int32)
    n_obs = host.integers(case["obs_min"], case["obs_max"] + 1, n).astype(np.int64)
    obs_off = np.concatenate([[0], np.cumsum(n_obs)]).astype(np.int64)
    J = torch.as_tensor(n_pl, device="cuda").long()
    counts = torch.as_tensor(n_obs, device="cuda")
    sys_of = torch.repeat_interleave(torch.arange(n, device="cuda"), counts)
    total = int(obs_off[-1])
    # times in order within each system: sort the pairs (system, time)
    span = _uniform(gen, (n,), 500.0, 6000.0)
    t = EPOCH + torch.sort(sys_of + _uniform(gen, (total,), 0.0, 1.0)).values.sub_(sys_of) \
        .clamp_(0.0, 1.0) * span[sys_of]
    sigma = _uniform(gen, (total,), 1.0, 5.0)
    planets = _planets(gen, n, top, case["e_max"])
    rows = torch.cat([planets.reshape(n, 5 * top), _uniform(gen, (n, 1), -10.0, 10.0)], dim=1)
    model = _scatter(gen, rows, top, case["perturb"])
    v = rows[:, -1][sys_of] + sigma * _normal(gen, (total,))
    for j in range(top):
        at = torch.nonzero(J[sys_of] > j).squeeze(1)
        for part in at.split(CHUNK):
            s = sys_of[part]
            v[part] += _velocity(*(planets[s, j, i] for i in range(5)), t[part])
    col = torch.arange(5 * top + 1, device="cuda")
    kept = (col[None, :] < 5 * J[:, None]) | (col[None, :] == 5 * top)
    return dict(obs_off=obs_off, n_pl=n_pl, params=model[kept], model=model, kept=kept, J=J,
                sys_of=sys_of, t=t, v=v, sigma=sigma)


def _kepler_inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = torch.float64 if case["mode"] == "fp64" else torch.float32
    # short of +-pi, where E jumps by 2 pi
    M = _uniform(gen, (case["n"],), -3.141592, 3.141592).to(kind)
    e = _uniform(gen, (case["n"],), 0.0, case["e_max"]).to(kind)
    return M, e


def prepare(case, seed):
    if case["kind"] == "kepler":
        M, e = _kepler_inputs(case, seed)
        return dict(case=case, M=M, e=e)
    if case["kind"] == "ragged":
        x = _ragged_inputs(case, seed)
        plan = kc.RaggedPlan(x["obs_off"], x["n_pl"], mode=case["mode"], want_grad=case["grad"])
        plan.set_observations(x["t"], x["v"], x["sigma"])
        return dict(case=case, plan=plan, params=x["params"])
    params, t, v, sigma = _uniform_inputs(case, seed)
    return dict(case=case, params=params, t=t, v=v, sigma=sigma)


# ------------------------------------------------------------ one pass

def run(state):
    case = state["case"]
    kind, mode = case["kind"], case["mode"]
    if kind == "kepler":
        return kc.kc_kepler_solve(state["M"], state["e"], mode=mode)
    if kind == "ragged":
        return state["plan"].run(state["params"])
    params, t, v, sigma = state["params"], state["t"], state["v"], state["sigma"]
    if kind == "predict":
        return kc.kc_rv_predict(params, t, t0=case["t0"])
    if kind == "chi2":
        if mode == "mixed" and case["t0"] == 0.0 and case["jitter"] == 0.0:
            return kc.kc_chi2_eval_mixed(params, t, v, sigma)
        if mode == "fp64" and case["t0"] == 0.0 and case["jitter"] == 0.0:
            return kc.kc_chi2_eval(params, t, v, sigma)
        return kc.kc_chi2_eval_ex(params, t, v, sigma, t0=case["t0"], jitter=case["jitter"],
                                  mode=mode)
    if kind == "grad":
        return kc.kc_chi2_grad(params, t, v, sigma, t0=case["t0"], jitter=case["jitter"],
                               mode=mode)
    if kind == "gn":
        return kc.kc_chi2_gauss_newton(params, t, v, sigma, t0=case["t0"], jitter=case["jitter"],
                                       mode=mode)
    p = params.detach().requires_grad_()
    if kind == "chi2_backward":
        value = kc.chi2(p, t, v, sigma, t0=case["t0"], jitter=case["jitter"], mode=mode)
    else:
        value = kc.nll(p, t, v, sigma, t0=case["t0"], mode=mode)
    value.sum().backward()
    return value.detach(), p.grad


# ------------------------------------------------------------ the work

# Floating-point operations (an FMA is two) of one planet-observation
# evaluation: phase, start, sine and cosine, one step of the solver and the
# velocity; and of its five derivatives with their sums.
FLOPS_EVAL, FLOPS_SOLVE, FLOPS_PARTIALS = 80.0, 60.0, 40.0


def _evals(case):
    if case["kind"] == "ragged":
        return case["n_sys"] * 3.5 * 0.5 * (case["obs_min"] + case["obs_max"])
    return float(case["n_sys"]) * case["n_pl"] * case["n_obs"]


def work(case):
    kind, out = case["kind"], 8 if case["mode"] == "fp64" else 4
    if kind == "kepler":
        return dict(bytes=3.0 * out * case["n"], flops=FLOPS_SOLVE * case["n"])
    evals = _evals(case)
    if kind == "ragged":
        n_par = case["n_sys"] * (5 * 3.5 + 1)
        obs = case["n_sys"] * 0.5 * (case["obs_min"] + case["obs_max"])
        return dict(bytes=8 * n_par + 24 * obs + out * (case["n_sys"] + case["grad"] * n_par),
                    flops=evals * (FLOPS_EVAL + case["grad"] * FLOPS_PARTIALS))
    n = 5 * case["n_pl"] + 1 + (kind == "nll_backward")
    S, N = case["n_sys"], case["n_obs"]
    read = 8.0 * S * n + 24.0 * N
    if kind == "predict":
        return dict(bytes=8.0 * S * n + 8.0 * N + 8.0 * S * N, flops=FLOPS_EVAL * evals)
    if kind == "chi2":
        return dict(bytes=read + out * S, flops=FLOPS_EVAL * evals)
    flops = (FLOPS_EVAL + FLOPS_PARTIALS) * evals
    if kind == "gn":
        tri = n * (n + 1) // 2
        return dict(bytes=read + out * S * (1 + n + tri), flops=flops + 2.0 * tri * S * N)
    grad = out * S * n if kind == "grad" else 8.0 * S * n      # autograd's is float64
    return dict(bytes=read + out * S + grad, flops=flops)


# ------------------------------------------------------------ 64 bits

def _exact_uniform(case, seed):
    params, t, v, sigma = _uniform_inputs(case, seed)
    kind, n_pl, t0 = case["kind"], case["n_pl"], case["t0"]
    dt = (t - t0)[None, :]
    S, N = case["n_sys"], case["n_obs"]
    got = []
    for p in params.split(max(1, CHUNK // (4 * N))):
        planet = [[p[:, 5 * j + i:5 * j + i + 1] for i in range(5)] for j in range(n_pl)]
        if kind in ("chi2", "predict"):
            V = p[:, 5 * n_pl:5 * n_pl + 1] + sum(_velocity(*q, dt) for q in planet)
            if kind == "predict":
                got.append((V,))
            else:
                got.append((((V - v) ** 2 / (sigma ** 2 + case["jitter"] ** 2)).sum(1),))
            continue
        V = p[:, 5 * n_pl:5 * n_pl + 1].expand(-1, N)
        cols = []
        for q in planet:
            vj, d = _partials(*q, dt)
            V = V + vj
            cols += list(d)
        r = V - v
        free = kind == "nll_backward"
        sj = p[:, 5 * n_pl + 1:5 * n_pl + 2] if free else case["jitter"]
        var = sigma ** 2 + sj ** 2
        w = 1.0 / var
        a = (w * r if free else 2.0 * w * r).expand(-1, N)
        g = [(a * d).sum(1) for d in cols] + [a.sum(1)]
        if free:
            value = 0.5 * (w * r * r + torch.log(TWO_PI * var)).sum(1)
            g.append((sj * w * (1.0 - w * r * r)).sum(1))
        else:
            value = (w * r * r).sum(1)
        out = [value, torch.stack(g, 1)]
        if kind == "gn":
            U = torch.stack([d.expand(-1, N) for d in cols] + [torch.ones_like(r)], 1) \
                * torch.sqrt(w)
            H = U @ U.transpose(1, 2)
            iu = torch.triu_indices(U.shape[1], U.shape[1], device=H.device)
            out.append(H[:, iu[0], iu[1]])
        got.append(tuple(out))
    cat = tuple(torch.cat(x) for x in zip(*got))
    return cat[0] if len(cat) == 1 else cat


def _exact_ragged(case, seed):
    x = _ragged_inputs(case, seed)
    sys_of, t, J, model, n = x["sys_of"], x["t"], x["J"], x["model"], case["n_sys"]
    V = model[:, -1][sys_of]
    for j in range(MAX_PLANETS_RAGGED):
        for part in torch.nonzero(J[sys_of] > j).squeeze(1).split(CHUNK):
            s = sys_of[part]
            V[part] += _velocity(*(model[s, 5 * j + i] for i in range(5)), t[part])
    w = 1.0 / x["sigma"] ** 2
    r = V - x["v"]

    def per_system(values, rows):
        return torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, rows, values)

    chi2 = per_system(w * r * r, sys_of)
    if not case["grad"]:
        return chi2
    g = torch.zeros_like(model)
    a = 2.0 * w * r
    g[:, -1] = per_system(a, sys_of)
    for j in range(MAX_PLANETS_RAGGED):
        for part in torch.nonzero(J[sys_of] > j).squeeze(1).split(CHUNK):
            s = sys_of[part]
            _, d = _partials(*(model[s, 5 * j + i] for i in range(5)), t[part])
            for i in range(5):
                g[:, 5 * j + i] += per_system(a[part] * d[i], s)
    return chi2, g[x["kept"]]


def exact(case, seed):
    if case["kind"] == "kepler":
        M, e = (x.double() for x in _kepler_inputs(case, seed))
        return torch.cat([_eccentric(m, k) for m, k in zip(M.split(CHUNK), e.split(CHUNK))])
    return (_exact_ragged if case["kind"] == "ragged" else _exact_uniform)(case, seed)
