"""The mixed path outside day-scaled inputs: periods down to seconds, spans of
10^6 days, times and periods given in seconds, with planets of both kinds in a
system.  The phase keeps pair-of-single precision there: chi2 within 1e-5
max(chi2, 1) plus the residuals' rounding carried into chi2, gradients and
normal matrices within the parity tests' bounds (tests/tolerance.py)."""
import numpy as np
import pytest
import torch
from test_gpu_pair import rows
from tolerance import (U32, chi2_rounding_term, grad_excess, grad_excess_ragged, ragged_ariths,
                       uniform_arith)

pytestmark = pytest.mark.gpu

DAY = 86400.0
# (name, first time, period range, span, other planets' period range, n_obs)
FORMS = {
    "milliday": (0.0, (1e-3, 2e-3), 4000.0, (1.0, 3000.0), 130),
    "seconds_of_period": (0.0, (1e-5, 1.2e-5), 40.0, (0.5, 3.0), 97),
    "far": (2450000.0, (1000.0, 3000.0), 1e6, (300.0, 9000.0), 256),
    "far_and_short": (2450000.0, (0.5, 2.0), 1e6, (1000.0, 3000.0), 129),
    "in_seconds": (2450000.0 * DAY, (DAY, 4000.0 * DAY), 4000.0 * DAY, (DAY, 4000.0 * DAY), 256),
    "last_tile_far": (2450000.0, (2.0, 900.0), 3000.0, (2.0, 900.0), 1300),
}


@pytest.fixture(scope="module")
def kc():
    import paper_0812_2976_gb300 as kc
    from paper_0812_2976_gb300 import build
    build.build()
    kc._lib.load()
    return kc


def batch(oracle_mod, form, n_sys, n_pl, seed=1):
    """Models at the truth up to one part in 1e7 of every other parameter than
    the periods, so that chi2 is about n_obs and its error shows the phase's."""
    epoch, p_range, span, other, n_obs = FORMS[form]
    rng = np.random.default_rng(seed)
    par = rows(rng, n_sys, n_pl, p_range, (0.0, 0.8))
    if n_pl > 1:
        par[:, 5:-1:5] = rows(rng, n_sys, n_pl - 1, other, (0.0, 0.8))[:, 0:-1:5]
    par[1:, 0:-1:5] = par[0, 0:-1:5]
    for i in (1, 2, 3, 4, 5):
        par[1:, i::5] = par[0, i::5] * (1.0 + 1e-7 * rng.standard_normal(par[1:, i::5].shape))
    t = np.sort(rng.uniform(epoch, epoch + span, n_obs))
    if form == "last_tile_far":
        t[1100:] += 60000.0
    sig = rng.uniform(1.0, 4.0, n_obs)
    v = oracle_mod.predict(par[:1], t, n_pl, epoch)[0] + sig * rng.standard_normal(n_obs)
    return par, t, v, sig, epoch


def chi2_bound(oracle_mod, par, t, v, sig, n_pl, epoch, ref):
    return 1e-5 * np.maximum(ref, 1.0) + chi2_rounding_term(oracle_mod, par, t, v, sig, n_pl,
                                                            epoch, 0.0, U32)


@pytest.mark.parametrize("n_pl", [1, 4])
@pytest.mark.parametrize("form", FORMS)
def test_chi2(kc, oracle_mod, form, n_pl):
    par, t, v, sig, epoch = batch(oracle_mod, form, 130, n_pl)
    ref = oracle_mod.chi2(par, t, v, sig, n_pl, t0=epoch)
    args = [torch.tensor(x, device="cuda") for x in (par, t, v, sig)]
    got, resid = kc.kc_chi2_eval_ex(*args, t0=epoch, mode="mixed", max_kepler_resid=True)
    got = got.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - ref) <= chi2_bound(oracle_mod, par, t, v, sig, n_pl, epoch, ref))
    assert float(resid.max()) <= 4e-6


@pytest.mark.parametrize("n_pl", [1, 3])
@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("what", ["grad", "gn0", "gn4"])
def test_gradient_and_normal_matrix(kc, oracle_mod, form, n_pl, what):
    par, t, v, sig, epoch = batch(oracle_mod, form, 90, n_pl)
    n_obs = t.size
    ref, gref, gabs = oracle_mod.chi2(par, t, v, sig, n_pl, t0=epoch, gabs=True)
    args = [torch.tensor(x, device="cuda") for x in (par, t, v, sig)]
    if what == "grad":
        chi2, grad = kc.kc_chi2_grad(*args, t0=epoch, mode="mixed")
        ar = uniform_arith(kc, oracle_mod, par, t, v, sig, n_pl, epoch, 0.0, "mixed")
    else:
        kc.kc_set_tile("gn", "mixed", 90, n_pl, n_obs, (32, 128, int(what[2])))
        try:
            chi2, grad, H = kc.kc_chi2_gauss_newton(*args, t0=epoch)
        finally:
            kc.kc_set_tile("gn", "mixed", 90, n_pl, n_obs, None)
        ar = uniform_arith(kc, oracle_mod, par, t, v, sig, n_pl, epoch, 0.0, "mixed", "gn")
        n = 5 * n_pl + 1
        Hr = oracle_mod.unpack_symmetric(oracle_mod.gauss_newton(par, t, sig, n_pl, t0=epoch), n)
        Hg = oracle_mod.unpack_symmetric(H.cpu().numpy().astype(np.float64), n)
        d = np.sqrt(np.diagonal(Hr, axis1=1, axis2=2))
        assert np.max(np.abs(Hg - Hr) / (d[:, :, None] * d[:, None, :])) <= 1e-4
    got = chi2.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - ref) <= chi2_bound(oracle_mod, par, t, v, sig, n_pl, epoch, ref))
    assert grad_excess(grad.cpu().numpy(), gref, gabs, 1e-3, U32, ar) <= 1.0


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("grad", [False, True])
def test_ragged(kc, oracle_mod, form, grad):
    """Systems of 1, 2 and 3 planets, each with the form's own times."""
    n_pl = np.array([1, 2, 3] * 8, np.int32)
    parts = [batch(oracle_mod, form, 1, int(J), seed=s) for s, J in enumerate(n_pl)]
    epoch = parts[0][4]
    par, t, v, sig = (np.concatenate([np.ravel(x[i]) for x in parts]) for i in range(4))
    off = lambda sizes: np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)  # noqa: E731
    obs_off, par_off = off([x[1].size for x in parts]), off(5 * n_pl + 1)
    plan = kc.RaggedPlan(obs_off, n_pl, t0=epoch, mode="mixed", want_grad=grad)
    plan.set_observations(*(torch.tensor(x, device="cuda") for x in (t, v, sig)))
    out = plan.run(torch.tensor(par, device="cuda"))
    chi2 = (out[0] if grad else out).cpu().numpy()
    ref, gref, gabs = oracle_mod.chi2_ragged(par, par_off, n_pl, t, v, sig, obs_off, t0=epoch,
                                             gabs=True)
    for s, (p, ts, vs, ss, _) in enumerate(parts):
        bound = chi2_bound(oracle_mod, p, ts, vs, ss, int(n_pl[s]), epoch, ref[s:s + 1])[0]
        assert abs(float(chi2[s]) - ref[s]) <= bound
    if grad:
        ar = ragged_ariths(oracle_mod, par, par_off, n_pl, t, v, sig, obs_off, epoch, 0.0, "mixed")
        assert grad_excess_ragged(out[1].cpu().numpy(), gref, gabs, par_off, 1e-3, U32, ar) <= 1.0


# (P range, span, unit, epoch): circular orbits at two times, the first without weight,
# so that chi2 is (cos M + 2)^2 of the second
PHASES = {
    "ordinary": ((1.0, 3000.0), 4000.0, 1.0, 2450000.0),
    "ordinary_far": ((1.0, 3000.0), 5e4, 1.0, 2450000.0),
    "far": ((3000.0, 3010.0), 1e6, 1.0, 2450000.0),
    "farther": ((3000.0, 3010.0), 3.9e6, 1.0, 2450000.0),
    "half_day": ((0.45, 0.55), 4000.0, 1.0, 2450000.0),
    "hours": ((0.06, 0.07), 16000.0, 1.0, 0.0),
    "milliday": ((1e-3, 1.1e-3), 4000.0, 1.0, 0.0),
    "tenth_of_that": ((1e-4, 1.1e-4), 300.0, 1.0, 0.0),
    "second": ((1e-5, 1.1e-5), 40.0, 1.0, 0.0),
    "in_seconds": ((1.0, 3000.0), 4000.0, DAY, 2450000.0),
    "in_years": ((1.0, 3000.0), 4000.0, 1.0 / 365.25, 2450000.0),
}


@pytest.mark.parametrize("form", PHASES)
@pytest.mark.parametrize("what", ["chi2", "grad", "gn0", "gn4", "ragged"])
def test_error_of_the_mean_anomaly(kc, oracle_mod, form, what):
    """The error of V seen in chi2, rms over 2048 systems and six times: M's
    (KAPPA_M u at most, tests/tolerance.py), the solve's and the sine's 3 u each,
    the velocity's 4 u and chi2's 3 u, each uniform: in quadrature over sqrt(3)
    3.2e-7 (the lost digits gave 4.5e-7 to 2e-4)."""
    p_range, span, unit, epoch = PHASES[form]
    epoch *= unit
    rng = np.random.default_rng(17)
    n = 2048
    par = rows(rng, n, 1, p_range, (0.0, 0.0))
    par[:, 0] *= unit
    par[:, 1], par[:, 3], par[:, 5] = 1.0, 0.0, 0.0
    put = lambda x: torch.tensor(x, device="cuda")  # noqa: E731
    v, sig = np.array([0.0, -2.0]), np.array([np.inf, 1.0])
    errors = []
    for last in rng.uniform(0.5, 1.0, 6):
        t = epoch + np.array([0.0, last * span * unit])
        V = oracle_mod.predict(par, t, 1, epoch)[:, 1]
        if what == "chi2":
            got = kc.kc_chi2_eval_ex(put(par), put(t), put(v), put(sig), t0=epoch, mode="mixed")
        elif what == "grad":
            got = kc.kc_chi2_grad(put(par), put(t), put(v), put(sig), t0=epoch, mode="mixed")[0]
        elif what == "ragged":
            plan = kc.RaggedPlan(2 * np.arange(n + 1), np.ones(n, np.int32), t0=epoch,
                                 mode="mixed")
            plan.set_observations(*(put(np.tile(x, n)) for x in (t, v, sig)))
            got = plan.run(put(par.ravel()))
        else:
            kc.kc_set_tile("gn", "mixed", n, 1, 2, (32, 128, int(what[2])))
            try:
                got = kc.kc_chi2_gauss_newton(put(par), put(t), put(v), put(sig), t0=epoch)[0]
            finally:
                kc.kc_set_tile("gn", "mixed", n, 1, 2, None)
        errors.append((got.cpu().numpy() - (V + 2.0) ** 2) / (2.0 * (V + 2.0)))
    assert np.sqrt(np.mean(np.square(errors))) <= 3.2e-7
