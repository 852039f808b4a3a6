"""Double-precision chi2 and velocities at amplitudes of every
unit a caller may use, and beyond the range of single precision: relative
agreement with the oracle as at m/s (chi2 1e-12; velocities 1e-11 of the
amplitude's scale), also for planets of very different amplitudes."""
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


@pytest.mark.parametrize("unit", [1e-60, 1e-30, 1e-18, 3e-9, 1e6, 1e30, 1e45, 1e90])
@pytest.mark.parametrize("n_pl", [1, 3])
def test_amplitudes(kc, oracle_mod, unit, n_pl):
    rng = np.random.default_rng(4)
    n_sys, n_obs = 50, 90
    par = rows(rng, n_sys, n_pl, (2.0, 900.0), (0.0, 0.9))
    par[:, 1:-1:5] *= unit
    par[:, -1] *= unit
    par[::5, 1] = 0.0                                  # no amplitude at all
    if n_pl > 1:
        par[1::5, 6] *= 1e-9                           # and one far below the others
    t = np.sort(rng.uniform(T0, T0 + 3000.0, n_obs))
    sig = unit * rng.uniform(1.0, 4.0, n_obs)
    v = oracle_mod.predict(par[1:2], t, n_pl, T0)[0] + sig * rng.standard_normal(n_obs)
    ref = oracle_mod.chi2(par, t, v, sig, n_pl, t0=T0)
    model = oracle_mod.predict(par, t, n_pl, T0)
    x = [torch.tensor(a, device="cuda") for a in (par, t, v, sig)]
    got = kc.kc_chi2_eval_ex(*x, t0=T0, mode="fp64").cpu().numpy()
    assert np.max(np.abs(got - ref) / np.maximum(ref, 1.0)) <= 1e-12
    vel = kc.kc_rv_predict(x[0], x[1], t0=T0).cpu().numpy()
    assert np.max(np.abs(vel - model)) <= 1e-11 * 50.0 * unit * n_pl / 0.1
