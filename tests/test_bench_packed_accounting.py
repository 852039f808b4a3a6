"""The benchmark's roofline numerators of the packed kernels and of the FP64 chi2:
FLOPs per planet-observation evaluation, operation by operation as kc_pair.cuh
and kc_f64.cuh write them (no GPU needed; FMA = 2, add / mul = 1, negations,
MUFU and integer operations 0).  A change to a count that the kernels did not
make fails here."""
import pytest

import bench

FMA, ADD, MUL = 2, 1, 1

# mean_anomaly_pair: y; k (two additions); u; the low parts; M
MEAN_ANOMALY = FMA + 2 * ADD + (FMA + ADD) + 2 * FMA + FMA
# kepler_pair: b, w; start_root (sum, a third, difference); x; the quartic; E0
START = MUL + FMA + (ADD + MUL + ADD) + MUL + 4 * FMA + FMA
# k; d0 (two differences); h0; s0 and c0 to second order
SIN_COS = ADD + 2 * ADD + MUL + 2 * FMA + 2 * FMA
# f; 1 - e cos E; d; h; sin and cos of the root
NEWTON = (ADD + FMA) + FMA + MUL + MUL + 2 * FMA + 2 * FMA
# velocity_sum: D; the numerator; the quotient inside the sum's first operation;
# the compensated sum's other three
VELOCITY = FMA + (MUL + FMA) + FMA + 3 * ADD
# per observation: the residual of two float pairs, its weighted square and the
# compensated sum
RESIDUAL = 3 * ADD + 2 * MUL + 4 * ADD


@pytest.mark.parametrize("n_pl", [1, 4, 8])
def test_packed_chi2_flops(n_pl):
    per_planet = MEAN_ANOMALY + START + SIN_COS + NEWTON + VELOCITY
    assert per_planet == 67 and RESIDUAL == 9
    assert bench.pair_flops_per_eval(n_pl) == per_planet + RESIDUAL / n_pl
    assert bench.chi2_flops_per_eval(n_pl, (32, 864, 3)) == bench.pair_flops_per_eval(n_pl)
    assert bench.chi2_flops_per_eval(n_pl, (32, 256, 0)) == bench.mixed_flops_per_eval(n_pl)


@pytest.mark.parametrize("n_pl", [1, 3, 8])
def test_packed_adjoint_flops(n_pl):
    # 1 - cos E from its own table: cos E beside it at the table's angle and at the start
    solve = MEAN_ANOMALY + START + SIN_COS + NEWTON + 2 * ADD
    # grad_terms: D; dK and Q of three operations each; K dK inside the compensated
    # sum, whose other operations are three additions
    terms = FMA + (2 * FMA + MUL) + (2 * FMA + MUL) + FMA + 3 * ADD
    # grad_add: Q y, Q y^2; beta y + 1/beta; the compensated period column; K;
    # e (two products and the sum); w; M
    sums = 2 * MUL + FMA + (FMA + 3 * ADD) + FMA + (2 * MUL + FMA) + FMA + FMA
    # per observation: the residual, w r, 2 w r, chi2's product and compensated
    # sum, gamma's sum, 2 w r (t - t0)
    per_obs = 3 * ADD + MUL + ADD + (MUL + 4 * ADD) + ADD + MUL
    assert (solve, terms, sums, per_obs) == (59, 17, 19, 12)
    assert bench.pair_grad_flops_per_eval(n_pl) == solve + terms + sums + per_obs / n_pl
    row = 5 + 1.0 / n_pl                    # sqrt(w) J, per planet and per observation
    adjoint = bench.pair_grad_flops_per_eval if n_pl <= 3 else bench.grad_flops_per_eval
    assert bench.gauss_newton_flops_per_eval(n_pl) == adjoint(n_pl) + row


@pytest.mark.parametrize("n_pl", [1, 4])
def test_fp64_float_expansion_flops(n_pl):
    # FP64 only: the phase (FMA, addition); f(E) (two FMAs); the velocity at the
    # table's angle (product, FMA) and its quotient into the sum (FMA); per
    # observation gamma - v, the corrections' addition, the weighted square
    assert bench.f64_flops_per_eval(n_pl) == ((FMA + ADD) + 2 * FMA + (MUL + FMA + FMA)
                                              + (ADD + ADD + MUL + FMA) / n_pl)
