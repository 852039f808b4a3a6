"""A time that is no number, or infinite, at the first observation (the
reference time of all others) or in the middle: the double-precision results
that depend on it are NaN, below and above e = 0.95, and the systems are
counted."""
import numpy as np
import pytest
import torch
from test_gpu_pair import T0, rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kc():
    import paper_0812_2976_gb300 as kc
    from paper_0812_2976_gb300 import build
    build.build()
    kc._lib.load()
    return kc


def put(*arrs):
    return [torch.tensor(a, device="cuda") for a in arrs]


N_SYS, N_OBS = 40, 70


def batch(n_pl, e_range, at, bad):
    rng = np.random.default_rng(3)
    par = rows(rng, N_SYS, n_pl, (2.0, 900.0), e_range)
    t = np.sort(rng.uniform(T0, T0 + 3000.0, N_OBS))
    t[at] = bad
    return par, t, np.zeros(N_OBS), np.ones(N_OBS)


@pytest.mark.parametrize("at", [0, 33])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, 1e60])
@pytest.mark.parametrize("n_pl,e_range", [(1, (0.0, 0.5)), (3, (0.5, 0.94)), (2, (0.0, 0.99))])
def test_double_precision_results_are_nan(kc, n_pl, e_range, bad, at):
    par, t, v, s = batch(n_pl, e_range, at, bad)
    x = put(par, t, v, s)
    kc.kc_last_device_error()
    assert torch.isnan(kc.kc_chi2_eval_ex(*x, t0=T0, mode="fp64")).all()
    assert kc.kc_last_device_error() == N_SYS
    chi2, grad = kc.kc_chi2_grad(*x, t0=T0, mode="fp64")
    assert torch.isnan(chi2).all() and torch.isnan(grad).all()
    assert kc.kc_last_device_error() == N_SYS
    free, = put(np.concatenate([par, np.ones((N_SYS, 1))], axis=1))
    assert torch.isnan(kc.kc_nll_eval(free, *x[1:], t0=T0, mode="fp64")).all()
    nll, grad = kc.kc_nll_grad(free, *x[1:], t0=T0, mode="fp64")
    assert torch.isnan(nll).all() and torch.isnan(grad).all()
    kc.kc_last_device_error()
    # velocities: at every time where the reference time is bad, else at that time
    # (a finite reference time is at no distance from itself)
    want = np.arange(N_OBS) == at
    if at == 0:
        want = ~want if np.isfinite(bad) else np.ones(N_OBS, bool)
    got = torch.isnan(kc.kc_rv_predict(x[0], x[1], t0=T0)).cpu().numpy()
    assert np.array_equal(got, np.tile(want, (N_SYS, 1)))
    got = torch.isnan(kc.kc_rv_predict_ragged(
        x[0].reshape(-1), torch.arange(N_SYS, device="cuda") * (5 * n_pl + 1),
        torch.full((N_SYS,), n_pl, device="cuda"), x[1].repeat(N_SYS),
        torch.arange(N_SYS + 1, device="cuda") * N_OBS, t0=T0)).cpu().numpy()
    assert np.array_equal(got, np.tile(want, N_SYS))
