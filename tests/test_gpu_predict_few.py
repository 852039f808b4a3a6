"""Model velocities at one to nine times: as many threads per system as there
are times (1 to 16), systems on both sides of a block's share, and more planets
than fit 48 KB of shared memory."""
import numpy as np
import pytest
import torch
from test_gpu_pair import T0, rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_obs", [1, 2, 3, 4, 5, 8, 9])
@pytest.mark.parametrize("n_sys,n_pl", [(1, 1), (127, 2), (129, 8), (1000, 5)])
def test_few_times(oracle_mod, n_sys, n_pl, n_obs):
    import paper_0812_2976_gb300 as kc
    rng = np.random.default_rng(n_sys + n_obs)
    par = rows(rng, n_sys, n_pl, (1.0, 4000.0), (0.0, 0.97))
    t = np.sort(rng.uniform(T0, T0 + 4000.0, n_obs))
    ref = oracle_mod.predict(par, t, n_pl, T0)
    got = kc.kc_rv_predict(torch.tensor(par, device="cuda"), torch.tensor(t, device="cuda"),
                           t0=T0).cpu().numpy()
    assert np.max(np.abs(got - ref)) <= 1e-11 * 50.0 * n_pl / 0.03
