"""A system's results do not depend on the systems it is evaluated with: the
bits of a row are the same beside rows of short periods, of phases past 1e5
periods and of e > 0.95 as beside ordinary ones, at the same launch shape; and
an element of a Kepler solve's beside elements that need the other solver, and
wherever it lies in memory."""
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


def two_batches(n_pl, p_range, e_range, plain=(1.0, 3000.0), n_sys=512, n_obs=200):
    """Rows of which every third is ordinary in both batches; the others are
    ordinary in the first and drawn from the given ranges in the second."""
    rng = np.random.default_rng(n_pl)
    plain = rows(rng, n_sys, n_pl, plain, (0.0, 0.93))
    mixed = plain.copy()
    odd = np.arange(n_sys) % 3 != 0
    mixed[odd] = rows(rng, int(odd.sum()), n_pl, p_range, e_range)
    t = np.sort(rng.uniform(T0, T0 + 4000.0, n_obs))
    v, s = rng.normal(0.0, 30.0, n_obs), rng.uniform(1.0, 4.0, n_obs)
    put = lambda x: torch.tensor(x, device="cuda")  # noqa: E731
    return put(plain), put(mixed), [put(x) for x in (t, v, s)], ~torch.tensor(odd)


ODD = [((0.004, 0.02), (0.0, 0.9), (0.05, 0.1)),      # 1e5 periods and more; up to 8e4
       ((1.0, 3000.0), (0.951, 0.99), (1.0, 3000.0))]


@pytest.mark.parametrize("p_range,e_range,ordinary", ODD)
@pytest.mark.parametrize("n_pl", [1, 3, 5])
def test_double_precision(kc, n_pl, p_range, e_range, ordinary):
    plain, mixed, obs, same = two_batches(n_pl, p_range, e_range, ordinary)
    for kernel in ("chi2", "grad"):
        kc.kc_set_tile(kernel, "fp64", 512, n_pl, 200, (4, 64))
    try:
        for fn in (lambda p: (kc.kc_chi2_eval_ex(p, *obs, t0=T0, mode="fp64"),),
                   lambda p: kc.kc_chi2_grad(p, *obs, t0=T0, mode="fp64"),
                   lambda p: (kc.kc_rv_predict(p, obs[0][:9].contiguous(), t0=T0),)):
            for a, b in zip(fn(plain), fn(mixed)):
                assert torch.equal(a.cpu()[same], b.cpu()[same])
    finally:
        for kernel in ("chi2", "grad"):
            kc.kc_set_tile(kernel, "fp64", 512, n_pl, 200, None)


@pytest.mark.parametrize("n_pl", [1, 3])
@pytest.mark.parametrize("split", [0, 4])
def test_mixed_short_periods(kc, n_pl, split):
    plain, mixed, obs, same = two_batches(n_pl, (0.01, 0.4), (0.0, 0.9))
    kc.kc_set_tile("chi2", "mixed", 512, n_pl, 200, (8, 128, 3))
    kc.kc_set_tile("grad", "mixed", 512, n_pl, 200, (4, 128))
    kc.kc_set_tile("gn", "mixed", 512, n_pl, 200, (32, 128, split))
    try:
        for fn in (lambda p: (kc.kc_chi2_eval_ex(p, *obs, t0=T0, mode="mixed"),),
                   lambda p: kc.kc_chi2_grad(p, *obs, t0=T0, mode="mixed"),
                   lambda p: kc.kc_chi2_gauss_newton(p, *obs, t0=T0)):
            for a, b in zip(fn(plain), fn(mixed)):
                assert torch.equal(a.cpu()[same], b.cpu()[same])
    finally:
        for kernel in ("chi2", "grad", "gn"):
            kc.kc_set_tile(kernel, "mixed", 512, n_pl, 200, None)


@pytest.mark.parametrize("mode", ["fp64", "mixed"])
def test_kepler_solve(kc, mode):
    rng = np.random.default_rng(2)
    kind = np.float64 if mode == "fp64" else np.float32
    M = rng.uniform(-3.1, 3.1, 4096).astype(kind)
    e = rng.uniform(0.0, 0.94, 4096).astype(kind)
    M2, e2 = M.copy(), e.copy()
    e2[1::7], M2[3::7], e2[5::7] = 0.98, 1e-12, -0.0
    same = np.ones(4096, bool)
    same[1::7] = same[3::7] = same[5::7] = False
    a, b = (kc.kc_kepler_solve(torch.tensor(x, device="cuda"), torch.tensor(y, device="cuda"),
                               mode=mode).cpu().numpy() for x, y in ((M, e), (M2, e2)))
    assert np.array_equal(a[same], b[same])
    # nor on where in memory an element lies
    shifted = [torch.tensor(np.concatenate([[0], x]).astype(kind), device="cuda")[1:]
               for x in (M, e)]
    assert np.array_equal(kc.kc_kepler_solve(*shifted, mode=mode).cpu().numpy(), a)
    odd = [torch.tensor(x[:4093], device="cuda") for x in (M, e)]
    assert np.array_equal(kc.kc_kepler_solve(*odd, mode=mode).cpu().numpy(), a[:4093])
