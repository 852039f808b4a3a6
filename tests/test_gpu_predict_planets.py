"""Ragged model velocities of systems with any number of planets: the planet
counts are device data that no host check sees, so a count above the eight of
the batch evaluations is summed like any other."""
import numpy as np
import pytest
import torch
from test_gpu_pair import T0, rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("e_max", [0.9, 0.98])
def test_counts_around_and_above_eight(oracle_mod, e_max):
    import paper_0812_2976_gb300 as kc
    rng = np.random.default_rng(11)
    n_pl = np.array([1, 8, 9, 16, 7, 17, 32, 33, 8, 40] * 7)
    n_obs = rng.integers(1, 70, n_pl.size)
    par, t, ref = [], [], []
    for J, n in zip(n_pl, n_obs):
        p = rows(rng, 1, int(J), (1.0, 3000.0), (0.0, e_max))[0]
        ts = np.sort(rng.uniform(T0, T0 + 4000.0, n))
        # the oracle takes eight planets at a time, gamma once
        V = np.full(n, p[-1])
        for j in range(0, J, 8):
            q = np.append(p[5 * j:5 * min(J, j + 8)], 0.0)
            V += oracle_mod.predict(q[None, :], ts, (q.size - 1) // 5, T0)[0]
        par.append(p), t.append(ts), ref.append(V)
    # an invalid planet past the eighth makes its system NaN
    par[2][5 * 8 + 2] = 1.5
    off = lambda n: np.concatenate([[0], np.cumsum(n)]).astype(np.int64)  # noqa: E731
    put = lambda a: torch.tensor(a, device="cuda")  # noqa: E731
    got = kc.kc_rv_predict_ragged(put(np.concatenate(par)), put(off(5 * n_pl + 1)),
                                  put(n_pl.astype(np.int32)), put(np.concatenate(t)),
                                  put(off(n_obs)), t0=T0).cpu().numpy()
    start = off(n_obs)
    assert np.isnan(got[start[2]:start[3]]).all()
    for s, V in enumerate(ref):
        if s != 2:
            tol = 1e-11 * 50.0 * n_pl[s] / (1.0 - e_max)
            assert np.max(np.abs(got[start[s]:start[s + 1]] - V)) <= tol
