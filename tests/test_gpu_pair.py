"""The packed two-observation evaluation of the mixed path (kc_pair.cuh) at
the places where it changes form: periods on both sides of the short mean
anomaly's limit (0.5 d) and of 1/64 d, times beyond 2^14 and 2^17 days from the
first, eccentricities up to one float below 1, and observation counts around
the pairs, the chunks and the staged tile.  chi2 of every system against the
FP64 oracle within 1e-5 max(chi2, 1) plus the residuals' rounding carried
into chi2 (tests/tolerance.py)."""
import numpy as np
import pytest
import torch
from tolerance import U32, chi2_rounding_term, grad_excess, uniform_arith

pytestmark = pytest.mark.gpu

T0 = 2450000.0


@pytest.fixture(scope="module")
def kc():
    import paper_0812_2976_gb300 as kc
    from paper_0812_2976_gb300 import build
    build.build()
    kc._lib.load()
    return kc


def rows(rng, n_sys, n_pl, p_range, e_range):
    par = np.empty((n_sys, 5 * n_pl + 1))
    end = 5 * n_pl
    shape = (n_sys, n_pl)
    par[:, 0:end:5] = np.exp(rng.uniform(*np.log(p_range), shape))
    par[:, 1:end:5] = rng.uniform(1.0, 50.0, shape)
    par[:, 2:end:5] = rng.uniform(*e_range, shape)
    par[:, 3:end:5] = rng.uniform(0.0, 2 * np.pi, shape)
    par[:, 4:end:5] = rng.uniform(-np.pi, np.pi, shape)
    par[:, -1] = rng.uniform(-5.0, 5.0, n_sys)
    return par


FORMS = [
    ((0.50, 0.53), 4000.0, (0.0, 0.9), 3, 129),      # short form, every start of a period
    ((0.47, 0.4999), 4000.0, (0.0, 0.9), 2, 130),    # wide form just beyond it
    ((0.012, 0.02), 300.0, (0.0, 0.6), 2, 67),       # 1/P on both sides of 64 cycles/d
    ((2.0, 4000.0), 16380.0, (0.0, 0.95), 4, 255),   # |tau| up to 2^14 d
    ((2.0, 4000.0), 40000.0, (0.0, 0.95), 4, 255),   # beyond: the wide form
    ((50.0, 9000.0), 200000.0, (0.0, 0.8), 1, 96),   # beyond 2^17 d
    ((1.0, 4000.0), 4000.0, (0.0, 0.0), 2, 1),       # circular, a single observation
    ((1.0, 4000.0), 4000.0, (0.0, 0.95), 8, 3),
    ((1.0, 4000.0), 4000.0, (0.0, 0.95), 5, 1024),   # the staged tile, full
    ((1.0, 4000.0), 4000.0, (0.0, 0.95), 1, 1027),   # and beyond
]


@pytest.mark.parametrize("p_range,span,e_range,n_pl,n_obs", FORMS)
def test_chi2_where_the_form_changes(kc, oracle_mod, p_range, span, e_range, n_pl, n_obs):
    rng = np.random.default_rng(n_obs + n_pl)
    n_sys = 150
    par = rows(rng, n_sys, n_pl, p_range, e_range)
    t = np.sort(rng.uniform(T0, T0 + span, n_obs))
    sig = rng.uniform(1.0, 4.0, n_obs)
    v = oracle_mod.predict(par[:1], t, n_pl, T0)[0] + sig * rng.standard_normal(n_obs)
    ref = oracle_mod.chi2(par, t, v, sig, n_pl, t0=T0)
    bound = 1e-5 * np.maximum(ref, 1.0) + chi2_rounding_term(oracle_mod, par, t, v, sig, n_pl, T0,
                                                             0.0, U32)
    args = [torch.tensor(x, device="cuda") for x in (par, t, v, sig)]
    got = kc.kc_chi2_eval_ex(*args, t0=T0, mode="mixed").cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - ref) <= bound)


@pytest.mark.parametrize("lanes", [1, 8, 32])
@pytest.mark.parametrize("p_range,span,e_range,n_pl,n_obs", FORMS)
def test_gradient_where_the_form_changes(kc, oracle_mod, p_range, span, e_range, n_pl, n_obs,
                                         lanes):
    """chi2 as above, and every component of the gradient within the parity
    tests' bound (1e-3, plus the derived term where its sum cancels)."""
    rng = np.random.default_rng(100 + n_obs + n_pl)
    n_sys = 90
    par = rows(rng, n_sys, n_pl, p_range, e_range)
    t = np.sort(rng.uniform(T0, T0 + span, n_obs))
    sig = rng.uniform(1.0, 4.0, n_obs)
    v = oracle_mod.predict(par[:1], t, n_pl, T0)[0] + sig * rng.standard_normal(n_obs)
    ref, gref, gabs = oracle_mod.chi2(par, t, v, sig, n_pl, t0=T0, gabs=True)
    bound = 1e-5 * np.maximum(ref, 1.0) + chi2_rounding_term(oracle_mod, par, t, v, sig, n_pl, T0,
                                                             0.0, U32)
    args = [torch.tensor(x, device="cuda") for x in (par, t, v, sig)]
    kc.kc_set_tile("grad", "mixed", n_sys, n_pl, n_obs, (lanes, 64))
    try:
        chi2, grad = kc.kc_chi2_grad(*args, t0=T0, mode="mixed")
        ar = uniform_arith(kc, oracle_mod, par, t, v, sig, n_pl, T0, 0.0, "mixed")
    finally:
        kc.kc_set_tile("grad", "mixed", n_sys, n_pl, n_obs, None)
    assert np.all(np.abs(chi2.cpu().numpy().astype(np.float64) - ref) <= bound)
    assert grad_excess(grad.cpu().numpy(), gref, gabs, 1e-3, U32, ar) <= 1.0


def test_eccentricities_up_to_one(kc, oracle_mod):
    """e one double below 1 rounds to 1 in float: finite where the oracle is
    (away from pericentre), and the solve's residual within 4e-6 rad."""
    rng = np.random.default_rng(5)
    n_sys, n_obs = 64, 200
    par = rows(rng, n_sys, 1, (10.0, 900.0), (0.9, 0.999))
    par[:16, 2] = 1.0 - 2.0 ** -np.arange(10, 26)
    par[16, 2] = np.nextafter(1.0, 0.0)
    t = np.sort(rng.uniform(T0, T0 + 3000.0, n_obs))
    args = [torch.tensor(x, device="cuda")
            for x in (par, t, np.zeros(n_obs), np.ones(n_obs))]
    chi2, resid = kc.kc_chi2_eval_ex(*args, t0=T0, mode="mixed", max_kepler_resid=True)
    assert torch.isfinite(chi2).all()
    assert float(resid.max()) <= 4e-6


def test_times_and_parameters_out_of_range_stay_nan(kc):
    """A time or parameter that is no number makes its systems NaN and is
    looked up in the table by a masked index like any other."""
    rng = np.random.default_rng(6)
    par = rows(rng, 64, 2, (1.0, 100.0), (0.0, 0.9))
    par[3, 0], par[5, 2], par[7, 4], par[9, 0], par[11, 1] = -1.0, 1.0, np.nan, np.inf, np.inf
    t = np.sort(rng.uniform(T0, T0 + 3000.0, 100))
    v, s = np.zeros(100), np.ones(100)
    run = lambda tt: kc.kc_chi2_eval_ex(  # noqa: E731
        *[torch.tensor(x, device="cuda") for x in (par, tt, v, s)], t0=T0, mode="mixed").cpu()
    bad = torch.zeros(64, dtype=torch.bool)
    bad[[3, 5, 7, 9, 11]] = True
    assert torch.equal(torch.isnan(run(t)), bad)
    t[50] = np.nan
    assert torch.isnan(run(t)).all()
    kc.kc_last_device_error()                        # leaves the counter at zero


@pytest.mark.parametrize("split", [0, 4])
@pytest.mark.parametrize("n_pl,n_obs,n_sys,span", [
    (3, 600, 2600, 3000.0),        # several groups of systems per CTA, two staged tiles
    (2, 512, 5000, 3000.0),        # one full tile, staged once
    (1, 65, 9000, 30000.0),        # the wide mean anomaly
])
def test_gauss_newton_persistent(kc, oracle_mod, split, n_pl, n_obs, n_sys, span):
    """The pair forms of the Gauss-Newton kernel over several groups per CTA,
    sampled systems against the oracle: H within 1e-4 of the correlation
    scale, chi2 and gradient as in the other tests; an invalid system among
    those set up together."""
    rng = np.random.default_rng(n_obs + n_sys)
    par = rows(rng, n_sys, n_pl, (1.0, 3000.0), (0.0, 0.85))
    par[7, 2] = 1.5
    t = np.sort(rng.uniform(T0, T0 + span, n_obs))
    sig = rng.uniform(1.0, 4.0, n_obs)
    v = rng.normal(0.0, 30.0, n_obs)
    args = [torch.tensor(x, device="cuda") for x in (par, t, v, sig)]
    kc.kc_last_device_error()
    kc.kc_set_tile("gn", "mixed", n_sys, n_pl, n_obs, (32, 128, split))
    try:
        chi2, grad, H = [x.cpu().numpy().astype(np.float64)
                         for x in kc.kc_chi2_gauss_newton(*args, t0=T0)]
    finally:
        kc.kc_set_tile("gn", "mixed", n_sys, n_pl, n_obs, None)
    assert kc.kc_last_device_error() == 1 and np.isnan(chi2[7]) and np.isnan(H[7]).all()
    idx = np.setdiff1d(np.r_[0:12, rng.choice(n_sys, 60, replace=False), n_sys - 3:n_sys], [7])
    p = par[idx]
    ref, gref, gabs = oracle_mod.chi2(p, t, v, sig, n_pl, t0=T0, gabs=True)
    assert np.all(np.abs(chi2[idx] - ref) <= 1e-5 * np.maximum(ref, 1.0) + chi2_rounding_term(
        oracle_mod, p, t, v, sig, n_pl, T0, 0.0, U32))
    ar = uniform_arith(kc, oracle_mod, p, t, v, sig, n_pl, T0, 0.0, "mixed", "gn")
    assert grad_excess(grad[idx], gref, gabs, 1e-3, U32, ar) <= 1.0
    n = 5 * n_pl + 1
    Hr = oracle_mod.unpack_symmetric(oracle_mod.gauss_newton(p, t, sig, n_pl, t0=T0), n)
    Hg = oracle_mod.unpack_symmetric(H[idx], n)
    d = np.sqrt(np.diagonal(Hr, axis1=1, axis2=2))
    assert np.max(np.abs(Hg - Hr) / (d[:, :, None] * d[:, None, :])) <= 1e-4


@pytest.mark.parametrize("mode", ["mixed", "fp64"])
def test_backward_is_the_widened_product(kc, mode):
    """backward scales the kernel's gradient in float64: the bits of widening
    both factors first, under a strided incoming gradient, and differentiable
    by it."""
    rng = np.random.default_rng(5)
    par = torch.tensor(rows(rng, 33, 2, (2.0, 900.0), (0.0, 0.9)), device="cuda")
    t = torch.tensor(np.sort(rng.uniform(T0, T0 + 3000.0, 70)), device="cuda")
    v, sig = torch.zeros_like(t), torch.ones_like(t)
    p = par.clone().requires_grad_()
    value = kc.chi2(p, t, v, sig, t0=T0, mode=mode)
    g = torch.tensor(rng.standard_normal((33, 2)), device="cuda").to(value.dtype)[:, 0]
    g.requires_grad_()
    got, = torch.autograd.grad(value, p, g, create_graph=True)
    _, ref = kc._grad_call("kc_chi2_grad_scalar", par, t, v, sig, T0, 0.0, mode)
    assert got.dtype == torch.float64
    assert torch.equal(got, ref.double() * g.detach().double()[:, None])
    by_g, = torch.autograd.grad(got.sum(), g)
    want = ref.double().sum(dim=1)
    assert torch.allclose(by_g.double(), want, rtol=1e-5 if mode == "mixed" else 1e-12,
                          atol=1e-6 * float(want.abs().max()))
