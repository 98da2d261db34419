"""The likelihood kernels' covariance table itself, over smoothness and distance, against the oracle.

A prediction from one observed point with y = 1, sigma2 = 1 and no nugget is rho(d) exactly as the kernels read it.
Distances have at most eleven significant bits, so that u = (d / beta)^2 is exact in the kernels' float pair
and only the table is left.  Tolerances are those the covariance evaluator's table is held to: 4e-15 absolute,
2e-9 relative for d C / d beta, and 1e-8 relative where values are tiny (the plain FP32 tail of the
polynomials), down to correlations of 1e-27; beyond, where rho falls by half and more within an interval, 1e-4.
The smoothness values are those at which the oracle's Bessel product is good to that."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2403_07412_gb300 import datagen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_07412_gb300 import build, vecchia

    build.build()
    oracle.build()
    return vecchia


def _distances(lo, hi, count, seed):
    """Log-uniform, eleven significant bits."""
    g = datagen.rng(seed)
    d = np.exp(g.uniform(math.log(lo), math.log(hi), count))
    e = np.floor(np.log2(d)) - 10
    return np.round(d / 2.0**e) * 2.0**e


def _predicted(V, kernel, nu, d):
    plan = V.Plan(np.array([[0.0, 0.0], [65536.0, 0.0]]), 1, order=V.ORDER_RANDOM)
    plan.set_kernel(kernel)
    y = torch.ones(2, dtype=torch.float64, device="cuda")
    got = V.vecchia_predict(plan, np.stack([d, np.zeros_like(d)], 1), y, (1.0, 1.0, nu, 0.0))[0].cpu().numpy()
    plan.close()
    return got


def _check(got, want):
    err = np.abs(got - want)
    assert np.all(err <= 4e-15), err.max()
    rel = err / want
    tiny = want < 2.0**-7
    assert np.all(rel[tiny & (want > 1e-27)] <= 1e-8), rel[tiny & (want > 1e-27)].max()
    assert np.all(rel[tiny & (want > 1e-80)] <= 1e-4), rel[tiny & (want > 1e-80)].max()


@pytest.mark.parametrize("nu", [0.3, 0.5, 0.8, 1.0, 1.5, 2.0, 2.5, 3.7, 5.0])
def test_matern_values(V, nu):
    d = np.concatenate([_distances(2.0**-15, 4.0, 3000, 61), _distances(4.0, 180.0, 3000, 62)])
    want = oracle.matern(d, 1.0, 1.0, nu)
    assert (want < 1e-60).any()
    _check(_predicted(V, V.KERNEL_MATERN, nu, d), want)


@pytest.mark.parametrize("alpha", [0.4, 0.7, 1.0])
def test_power_exponential_values(V, alpha):
    d = np.concatenate([_distances(2.0**-15, 4.0, 3000, 63), _distances(4.0, 60.0, 3000, 64)])
    d = d[d**alpha < 180.0]
    _check(_predicted(V, V.KERNEL_POWEXP, alpha, d), oracle.powexp(d, 1.0, 1.0, alpha))


def test_beyond_the_table(V):
    """u >= 2^20 (the power exponential alone is not 0 there): FP64's own values, 0
    for those below its normal range."""
    d = _distances(1100.0, 5000.0, 200, 65)
    for alpha in (0.1, 0.4, 0.8):
        got, want = _predicted(V, V.KERNEL_POWEXP, alpha, d), np.exp(-(d**alpha))
        assert np.all(np.abs(got - want) <= 1e-11 * want + 2.3e-308)
    assert np.all(_predicted(V, V.KERNEL_MATERN, 1.5, d) == 0.0)


@pytest.mark.parametrize("nu", [0.3, 0.5, 1.0, 1.5, 2.37, 5.0])
def test_beta_gradient_of_a_pair(V, nu):
    """h through two locations, whose d l / d beta has a closed form, from strong correlation to 1e-13."""
    y, t2 = (0.75, -1.25), 0.5
    for x in _distances(2.0**-3, 30.0, 25, 66):
        one = np.array([x])
        rho, db = float(oracle.matern(one, 1.0, 1.0, nu)[0]), float(oracle.matern_dbeta(one, 1.0, 1.0, nu)[0])
        s, r = 1 + t2 - rho * rho / (1 + t2), y[1] - rho * y[0] / (1 + t2)
        ds, dr = -2 * rho * db / (1 + t2), -db * y[0] / (1 + t2)
        want = -r * dr / s + r * r * ds / (2 * s * s) - ds / (2 * s)
        plan = V.Plan(np.array([[0.0, 0.0], [x, 0.0]]), 1, order=V.ORDER_GIVEN, perm=np.arange(2))
        t = V.vecchia_loglik_terms(plan, torch.tensor(y, dtype=torch.float64, device="cuda"), (1.0, 1.0, nu, t2), want_grad=True)
        assert abs(float(t[1, 2]) - want) <= 2e-9 * abs(want), x
        plan.close()
