"""The mixed ragged kernel where its packed pairs and its queue can go wrong:
counts of 0 to 3 observations and around one and two rounds of a warp (64 and
128), short periods and far times (the wide mean anomaly) beside systems of the
short form, systems with an invalid planet among valid ones, and batches large
enough that a warp takes two, three or four systems at a time."""
import numpy as np
import pytest
import torch
from tolerance import U32, chi2_rounding_term, grad_excess_ragged, ragged_ariths

pytestmark = pytest.mark.gpu

T0 = 2450000.0
COUNTS = [0, 1, 2, 3, 5, 62, 63, 64, 65, 66, 127, 128, 129, 200]


@pytest.fixture(scope="module")
def kc():
    import paper_0812_2976_gb300 as kc
    from paper_0812_2976_gb300 import build
    build.build()
    kc._lib.load()
    return kc


@pytest.fixture(scope="module")
def batch(oracle_mod):
    """One system of each planet count and observation count, every third with
    a planet of P < 0.5 d, every fourth observed over 40000 d."""
    rng = np.random.default_rng(8)
    n_pl = np.repeat(np.arange(1, 9), len(COUNTS)).astype(np.int32)
    n_obs = np.tile(COUNTS, 8)
    order = rng.permutation(n_pl.size)
    n_pl, n_obs = n_pl[order], n_obs[order]
    obs_off = np.concatenate([[0], np.cumsum(n_obs)]).astype(np.int64)
    par_off = np.concatenate([[0], np.cumsum(5 * n_pl + 1)]).astype(np.int64)
    par, ts = [], []
    for s, J in enumerate(n_pl):
        P = np.exp(rng.uniform(np.log(2.0), np.log(4000.0), J))
        if s % 3 == 0:
            P[rng.integers(J)] = rng.uniform(0.3, 0.5)
        rows = np.stack([P, rng.uniform(1, 50, J), rng.uniform(0, 0.9, J),
                         rng.uniform(0, 2 * np.pi, J), rng.uniform(-np.pi, np.pi, J)], axis=1)
        par.append(np.append(rows.ravel(), rng.uniform(-5, 5)))
        ts.append(np.sort(rng.uniform(T0, T0 + (40000.0 if s % 4 == 0 else 4000.0), n_obs[s])))
    par, t = np.concatenate(par), np.concatenate(ts)
    sig = rng.uniform(1.0, 4.0, t.size)
    truth = par * (1.0 + 0.01 * rng.standard_normal(par.size))
    ecc = np.concatenate([np.append(np.tile([False, False, True, False, False], J), False)
                          for J in n_pl])
    truth[ecc] = np.minimum(truth[ecc], 0.95)
    v = oracle_mod.predict_ragged(truth, par_off, n_pl, t, obs_off, T0)
    return n_pl, par_off, par, obs_off, t, v + sig * rng.standard_normal(t.size), sig


def run(kc, n_pl, par, obs_off, t, v, sig, grad):
    put = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")
    plan = kc.RaggedPlan(obs_off, n_pl, t0=T0, mode="mixed", want_grad=grad)
    plan.set_observations(put(t), put(v), put(sig))
    out = plan.run(put(par))
    return [x.cpu().numpy() for x in (out if grad else (out,))]


@pytest.mark.parametrize("grad", [False, True])
def test_pairs_against_the_oracle(kc, oracle_mod, batch, grad):
    n_pl, par_off, par, obs_off, t, v, sig = batch
    out = run(kc, n_pl, par, obs_off, t, v, sig, grad)
    ref, gref, gabs = oracle_mod.chi2_ragged(par, par_off, n_pl, t, v, sig, obs_off, t0=T0,
                                             gabs=True)
    for s, J in enumerate(n_pl):
        o, p = slice(*obs_off[s:s + 2]), slice(*par_off[s:s + 2])
        extra = 0.0
        if o.stop > o.start:
            extra = chi2_rounding_term(oracle_mod, par[p], t[o], v[o], sig[o], int(J), T0, 0.0,
                                       U32)[0]
        assert abs(out[0][s] - ref[s]) <= 1e-5 * max(ref[s], 1.0) + extra, (s, out[0][s], ref[s])
    if grad:
        ar = ragged_ariths(oracle_mod, par, par_off, n_pl, t, v, sig, obs_off, T0, 0.0, "mixed")
        assert grad_excess_ragged(out[1], gref, gabs, par_off, 1e-3, U32, ar) <= 1.0


@pytest.mark.parametrize("grad", [False, True])
@pytest.mark.parametrize("copies", [175, 265, 350])
def test_company_changes_nothing(kc, batch, grad, copies):
    """Copies of the batch (19600, 29680 and 39200 systems: two, three and four
    taken at a time on 152 SMs), with an invalid eccentricity in every seventh
    system: the valid ones have the bits of the single batch, the others NaN."""
    n_pl, par_off, par, obs_off, t, v, sig = batch
    one = run(kc, n_pl, par, obs_off, t, v, sig, grad)
    bad = np.arange(n_pl.size * copies) % 7 == 3
    offs = lambda off: np.concatenate([[0], np.cumsum(np.tile(np.diff(off), copies))])
    many_off = offs(par_off)
    many = np.tile(par, copies)
    many[many_off[:-1][bad] + 2] = 1.0
    got = run(kc, np.tile(n_pl, copies), many, offs(obs_off), *(np.tile(x, copies)
                                                               for x in (t, v, sig)), grad)
    for k, single in enumerate(one):
        is_bad = bad if k == 0 else np.repeat(bad, np.tile(5 * n_pl + 1, copies))
        want = np.tile(single, copies)
        assert np.array_equal(got[k][~is_bad], want[~is_bad])
        assert np.all(np.isnan(got[k][is_bad]))
