"""The Kepler-only solvers where they change form: M at 0, next to the limits
2^-30 and pi and beyond 2 pi, e at 0, around 0.95 and next to 1, alone and
beside ordinary elements (a warp or a group of four takes one form together),
counts around the groups, and M and e that no solver takes."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

PI = np.pi
EDGE_M = [0.0, 1e-300, 1e-12, 2.0 ** -31, 2.0 ** -30, 2.0 ** -30 * (1 + 1e-9), 1e-4, 1.5, 3.14159,
          np.nextafter(PI, 0), PI - 1e-9, 3.5, 6.0, 7.0, 1e5]
EDGE_E = [0.0, 1e-9, 0.3, 0.9499, 0.95, 0.9500001, 0.96, 0.999]


@pytest.fixture(scope="module")
def kc():
    import paper_0812_2976_gb300 as kc
    from paper_0812_2976_gb300 import build
    build.build()
    kc._lib.load()
    return kc


def elements(n, ordinary, dtype):
    """n pairs: every edge M with every edge e and either sign, in an order
    that mixes them, `ordinary` of the elements replaced by plain ones."""
    rng = np.random.default_rng(n)
    M, e = (x.ravel() for x in np.meshgrid(np.concatenate([EDGE_M, -np.array(EDGE_M)]), EDGE_E))
    pick = rng.permutation(np.resize(np.arange(M.size), n))
    M, e = M[pick].astype(dtype), e[pick].astype(dtype)
    plain = rng.random(n) < ordinary
    M[plain] = rng.uniform(-3.1, 3.1, plain.sum())
    e[plain] = rng.uniform(0.0, 0.94, plain.sum())
    return M, e


def root(M, e):
    """E in extended precision on the branch of M reduced to [-pi, pi]."""
    M, e = M.astype(np.longdouble), e.astype(np.longdouble)
    two_pi = np.longdouble("6.283185307179586476925286766559")
    M = M - two_pi * np.rint(M / two_pi)
    m = np.abs(M)
    lo, hi = m.copy(), np.minimum(m + e, two_pi / 2)
    for _ in range(80):
        mid = (lo + hi) / 2
        up = mid - e * np.sin(mid) < m
        lo, hi = np.where(up, mid, lo), np.where(up, hi, mid)
    E = (lo + hi) / 2
    for _ in range(2):
        E = E - (E - e * np.sin(E) - m) / (1 - e * np.cos(E))
    return np.copysign(E, M), 1 - e * np.cos(E)


@pytest.mark.parametrize("n", [1, 3, 4, 31, 33, 1023, 4099])
@pytest.mark.parametrize("ordinary", [0.0, 0.97])
def test_edges(kc, n, ordinary):
    """Within 6 u max(|M|, pi) / (1 - e cos E), u the type's rounding: M's
    reduction (2 pi q rounded, q M's), E - M, sin E, e sin E and E are each
    rounded once, at most by u pi."""
    for mode, dtype, u in (("fp64", np.float64, 2.0 ** -53), ("mixed", np.float32, 2.0 ** -24)):
        M, e = elements(n, ordinary, dtype)
        E = kc.kc_kepler_solve(torch.tensor(M, device="cuda"), torch.tensor(e, device="cuda"),
                               mode=mode).cpu().numpy()
        ref, D = root(M, e)
        # M beyond pi: its reduction rounds 2 pi q
        reduced = np.maximum(np.abs(M.astype(np.float64)), PI)
        bound = 6 * u * reduced / D.astype(np.float64)
        diff = np.abs((E - ref).astype(np.float64))
        diff = np.minimum(diff, np.abs(diff - 2 * PI))       # +-pi are one angle
        assert np.all(diff <= bound), (mode, np.max(diff / bound))


@pytest.mark.parametrize("mode,dtype", [("fp64", torch.float64), ("mixed", torch.float32)])
def test_invalid_elements_stay_alone(kc, mode, dtype):
    """NaN and infinite M and NaN e give NaN; their neighbours stay roots."""
    M, e = (torch.tensor(x, device="cuda", dtype=dtype) for x in elements(1024, 1.0, np.float64))
    good = kc.kc_kepler_solve(M, e, mode=mode)
    M2, e2 = M.clone(), e.clone()
    M2[5::97], M2[11::131], e2[3::89] = float("nan"), float("inf"), float("nan")
    bad = torch.isnan(M2) | torch.isinf(M2) | torch.isnan(e2)
    E = kc.kc_kepler_solve(M2, e2, mode=mode)
    assert torch.isnan(E[bad]).all()
    tol = 64 * torch.finfo(dtype).eps
    assert (E[~bad] - good[~bad]).abs().max() <= tol
