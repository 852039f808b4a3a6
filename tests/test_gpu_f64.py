"""The FP64 evaluation in float expansions (kc_f64.cuh) where it can go wrong:
phases past 1e5 periods (the second wrap), eccentricities 0, on both sides of
0.95 within one warp and near the table's grid, pericentre and apocentre,
observation counts around the lanes and the staged tile, every planet count's
smallest launch; and model velocities around their chunk of observations.
FP64 tolerances of the parity tests: chi2 1e-12, gradient 1e-9 per component
(tests/tolerance.py), velocities 1e-11 of the largest amplitude's scale."""
import numpy as np
import pytest
import torch
from test_gpu_pair import T0, rows
from tolerance import U64, grad_excess, uniform_arith

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kc():
    import paper_0812_2976_gb300 as kc
    from paper_0812_2976_gb300 import build
    build.build()
    kc._lib.load()
    return kc


def dev(*arrs):
    return [torch.tensor(np.ascontiguousarray(a), device="cuda") for a in arrs]


@pytest.mark.parametrize("p_range,span,e_range,n_pl,n_obs", [
    ((0.01, 0.02), 4000.0, (0.0, 0.9), 2, 60),        # tau/P up to 4e5
    ((1.0, 4000.0), 4000.0, (0.0, 0.0), 1, 33),       # circular
    ((1.0, 4000.0), 4000.0, (0.93, 0.97), 3, 65),     # both solvers in a warp
    ((1.0, 4000.0), 4000.0, (0.0, 0.95), 8, 1),       # one observation
    ((1.0, 4000.0), 4000.0, (0.0, 0.95), 5, 127),
    ((300.0, 4000.0), 10.0, (0.0, 1e-9), 4, 31),      # phases within a few degrees
    ((1.0, 4000.0), 4000.0, (0.0, 0.95), 1, 2051),    # past the staged tile
])
@pytest.mark.parametrize("tile", [None, (1, 32), (32, 64)])
def test_chi2_and_gradient(kc, oracle_mod, p_range, span, e_range, n_pl, n_obs, tile):
    rng = np.random.default_rng(7 * n_obs + n_pl)
    n_sys = 70
    par = rows(rng, n_sys, n_pl, p_range, e_range)
    par[::7, 4] = 0.0                                # pericentre at the first time
    par[3::7, 4] = np.pi                             # apocentre
    t = np.sort(rng.uniform(T0, T0 + span, n_obs))
    t[0] = T0
    sig = rng.uniform(1.0, 4.0, n_obs)
    v = oracle_mod.predict(par[:1], t, n_pl, T0)[0] + sig * rng.standard_normal(n_obs)
    ref, gref, gabs = oracle_mod.chi2(par, t, v, sig, n_pl, t0=T0, gabs=True)
    args = dev(par, t, v, sig)
    for kernel in ("chi2", "grad"):
        kc.kc_set_tile(kernel, "fp64", n_sys, n_pl, n_obs, tile)
    try:
        got = kc.kc_chi2_eval_ex(*args, t0=T0, mode="fp64").cpu().numpy()
        chi2, grad = kc.kc_chi2_grad(*args, t0=T0, mode="fp64")
        ar = uniform_arith(kc, oracle_mod, par, t, v, sig, n_pl, T0, 0.0, "fp64")
    finally:
        for kernel in ("chi2", "grad"):
            kc.kc_set_tile(kernel, "fp64", n_sys, n_pl, n_obs, None)
    scale = np.maximum(ref, 1.0)
    assert np.max(np.abs(got - ref) / scale) <= 1e-12
    assert np.max(np.abs(chi2.cpu().numpy() - ref) / scale) <= 1e-12
    assert grad_excess(grad.cpu().numpy(), gref, gabs, 1e-9, U64, ar) <= 1.0


@pytest.mark.parametrize("n_sys,n_pl,n_obs", [(1, 1, 1), (3, 8, 7), (17, 2, 9), (40, 3, 128),
                                              (2, 4, 1025), (700, 1, 130)])
def test_model_velocities(kc, oracle_mod, n_sys, n_pl, n_obs):
    rng = np.random.default_rng(n_sys + n_obs)
    par = rows(rng, n_sys, n_pl, (1.0, 4000.0), (0.0, 0.97))
    t = np.sort(rng.uniform(T0, T0 + 4000.0, n_obs))
    ref = oracle_mod.predict(par, t, n_pl, T0)
    P, T = dev(par, t)
    got = kc.kc_rv_predict(P, T, t0=T0).cpu().numpy()
    assert np.max(np.abs(got - ref)) <= 1e-11 * 50.0 * n_pl / 0.03


def test_wide_tiles_of_many_planets_still_launch(kc, oracle_mod):
    """One thread per system in the largest block: the planets' constants
    alone take most of the shared memory (the gradient then runs smaller
    blocks)."""
    rng = np.random.default_rng(9)
    n_sys, n_pl, n_obs = 600, 8, 300
    par = rows(rng, n_sys, n_pl, (1.0, 4000.0), (0.0, 0.9))
    t = np.sort(rng.uniform(T0, T0 + 4000.0, n_obs))
    v, sig = rng.normal(0.0, 30.0, n_obs), rng.uniform(1.0, 4.0, n_obs)
    ref = oracle_mod.chi2(par, t, v, sig, n_pl, t0=T0)
    args = dev(par, t, v, sig)
    for kernel in ("chi2", "grad"):
        kc.kc_set_tile(kernel, "fp64", n_sys, n_pl, n_obs, (1, 256))
    try:
        got = [kc.kc_chi2_eval_ex(*args, t0=T0, mode="fp64"),
               kc.kc_chi2_grad(*args, t0=T0, mode="fp64")[0]]
    finally:
        for kernel in ("chi2", "grad"):
            kc.kc_set_tile(kernel, "fp64", n_sys, n_pl, n_obs, None)
    for x in got:
        assert np.max(np.abs(x.cpu().numpy() - ref) / np.maximum(ref, 1.0)) <= 1e-12
