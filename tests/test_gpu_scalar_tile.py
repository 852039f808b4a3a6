"""Autotuning the mixed gradient: the scalar kernel behind autograd and the
free-jitter likelihood is timed by itself and takes its own fastest shape, not
the one of the packed kernel."""
import re

import numpy as np
import torch
from test_gpu_pair import T0, rows
import pytest

pytestmark = pytest.mark.gpu


def test_each_kernel_takes_its_own_fastest_shape(capfd, monkeypatch):
    import paper_0812_2976_gb300 as kc
    rng = np.random.default_rng(1)
    n_sys, n_pl, n_obs = 3000, 2, 150
    args = [torch.tensor(x, device="cuda") for x in (
        rows(rng, n_sys, n_pl, (1.0, 3000.0), (0.0, 0.8)),
        np.sort(rng.uniform(T0, T0 + 4000.0, n_obs)), rng.normal(0.0, 30.0, n_obs),
        rng.uniform(1.0, 4.0, n_obs))]
    scalar = lambda: kc._grad_call("kc_chi2_grad_scalar", *args, T0, 0.0, "mixed")  # noqa: E731
    builtin = scalar()
    monkeypatch.setenv("KC_AUTOTUNE_VERBOSE", "1")
    try:
        tile, _ = kc.kc_autotune(*args, kernel="grad", mode="mixed")
        lines = re.findall(r"kind (\d) .* G +(\d+) block +(\d+) split 0: +([0-9.]+) us",
                           capfd.readouterr().err)
        times = {k: {(int(g), int(b)): float(us) for j, g, b, us in lines if j == k}
                 for k in "35"}
        assert set(times["5"]) == set(times["3"]) and len(times["5"]) > 10
        assert times["3"][tuple(tile[:2])] <= 1.02 * min(times["3"].values())
        tuned = scalar()
        fast = [t for t, us in times["5"].items() if us <= 1.02 * min(times["5"].values())]
        wanted = [builtin]
        for t in fast:
            kc.kc_set_tile("grad", "mixed", n_sys, n_pl, n_obs, t)
            wanted.append(scalar())
        assert any(all(torch.equal(x, y) for x, y in zip(tuned, w)) for w in wanted)
    finally:
        kc.kc_set_tile("grad", "mixed", n_sys, n_pl, n_obs, None)
    assert all(torch.equal(x, y) for x, y in zip(scalar(), builtin))
