"""Launches above 48 KB of dynamic shared memory next to launches that need
less of the same kernel: the limit a kernel was given for the larger one must
still hold after the smaller one, on one thread and on two."""
import threading

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kc():
    import paper_0812_2976_gb300 as kc
    from paper_0812_2976_gb300 import build
    build.build()
    kc._lib.load()
    return kc


def inputs(n_sys, n_pl, n_obs, seed):
    rng = np.random.default_rng(seed)
    par = np.empty((n_sys, 5 * n_pl + 1))
    par[:, 0:-1:5] = np.exp(rng.uniform(0.0, 8.0, (n_sys, n_pl)))
    par[:, 1:-1:5] = rng.uniform(1.0, 50.0, (n_sys, n_pl))
    par[:, 2:-1:5] = rng.uniform(0.0, 0.9, (n_sys, n_pl))
    par[:, 3:-1:5] = rng.uniform(0.0, 6.0, (n_sys, n_pl))
    par[:, 4:-1:5] = rng.uniform(-3.0, 3.0, (n_sys, n_pl))
    par[:, -1] = 0.0
    t = np.sort(rng.uniform(2450000.0, 2454000.0, n_obs))
    return [torch.tensor(x, device="cuda")
            for x in (par, t, rng.normal(0.0, 30.0, n_obs), rng.uniform(1.0, 4.0, n_obs))]


# (kernel, mode, n_pl, the larger and the smaller launch as (n_obs, tile)):
# 62336 and 51728 bytes; one thread per system in blocks of 256 and 128
CASES = [
    ("chi2", "mixed", 4, (1000, (8, 1024, 3)), (700, (8, 896, 3))),
    ("chi2", "fp64", 8, (300, (1, 256)), (600, (1, 128))),
    ("grad", "mixed", 8, (300, (1, 256)), (600, (1, 128))),
]


def calls(kc, kernel, mode, n_pl, shapes):
    out = []
    for n_obs, tile in shapes:
        x = inputs(300, n_pl, n_obs, n_obs)
        kc.kc_set_tile(kernel, mode, 300, n_pl, n_obs, tile)
        fn = kc.kc_chi2_grad if kernel == "grad" else kc.kc_chi2_eval_ex
        out.append(lambda x=x, fn=fn: fn(*x, t0=2450000.0, mode=mode)[0 if fn is kc.kc_chi2_grad
                                                                     else slice(None)])
    return out


def unset(kc, kernel, mode, n_pl, shapes):
    for n_obs, _ in shapes:
        kc.kc_set_tile(kernel, mode, 300, n_pl, n_obs, None)


@pytest.mark.parametrize("kernel,mode,n_pl,large,small", CASES)
def test_a_smaller_launch_leaves_the_limit(kc, kernel, mode, n_pl, large, small):
    shapes = (large, small)
    big, little = calls(kc, kernel, mode, n_pl, shapes)
    try:
        first, other = big(), little()
        for _ in range(2):
            assert torch.equal(big(), first)
            assert torch.equal(little(), other)
        assert torch.isfinite(first).all() and torch.isfinite(other).all()
    finally:
        unset(kc, kernel, mode, n_pl, shapes)


@pytest.mark.parametrize("kernel,mode,n_pl,large,small", CASES)
def test_two_threads_with_two_sizes(kc, kernel, mode, n_pl, large, small):
    """Each thread launches one of the sizes 2000 times; a limit lowered
    between another thread's setting and launch would fail the launch."""
    shapes = (large, small)
    failed = []

    def work(call):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(2000):
                    call()
        except Exception as err:  # noqa: BLE001 - reported by the assertion below
            failed.append(err)

    try:
        threads = [threading.Thread(target=work, args=(c,))
                   for c in calls(kc, kernel, mode, n_pl, shapes)]
        for th in threads:
            th.start()
        for th in threads:
            th.join()
        torch.cuda.synchronize()
    finally:
        unset(kc, kernel, mode, n_pl, shapes)
    assert not failed
