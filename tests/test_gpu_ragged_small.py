"""Ragged batches of systems with a handful of observations, at the sizes where a
warp takes one, two, three or four of them at a time (4864 systems for each on 152
SMs): the bits of a batch small enough for one, and the oracle's chi2."""
import numpy as np
import pytest
import torch
from test_gpu_pair import T0, rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grad", [False, True])
@pytest.mark.parametrize("copies", [24, 25, 49, 73, 98])
def test_bits_of_a_small_batch(oracle_mod, grad, copies):
    import paper_0812_2976_gb300 as kc
    rng = np.random.default_rng(6)
    n = 200
    n_pl = rng.integers(1, 9, n).astype(np.int32)
    n_obs = rng.integers(0, 18, n)
    par = np.concatenate([rows(rng, 1, int(J), (0.3, 3000.0), (0.0, 0.9))[0] for J in n_pl])
    t = np.concatenate([np.sort(rng.uniform(T0, T0 + 4000.0, k)) for k in n_obs])
    v, s = rng.normal(0.0, 30.0, t.size), rng.uniform(1.0, 4.0, t.size)
    put = lambda a: torch.tensor(a, device="cuda")  # noqa: E731

    def run(m):
        off = np.concatenate([[0], np.cumsum(np.tile(n_obs, m))]).astype(np.int64)
        plan = kc.RaggedPlan(off, np.tile(n_pl, m), t0=T0, mode="mixed", want_grad=grad)
        plan.set_observations(*(put(np.tile(x, m)) for x in (t, v, s)))
        out = plan.run(put(np.tile(par, m)))
        return [x.cpu().numpy() for x in (out if grad else (out,))]

    one, many = run(1), run(copies)
    for a, b in zip(one, many):
        assert np.array_equal(np.tile(a, copies), b)
    off = lambda k: np.concatenate([[0], np.cumsum(k)]).astype(np.int64)  # noqa: E731
    ref = oracle_mod.chi2_ragged(par, off(5 * n_pl + 1), n_pl, t, v, s, off(n_obs), t0=T0)
    assert np.max(np.abs(one[0] - ref) / np.maximum(ref, 1.0)) <= 1e-5
