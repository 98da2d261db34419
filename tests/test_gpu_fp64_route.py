"""Blocks of the fixed-point sizes that are eliminated in FP64 all the same: a few data that tower over the others,
a location barely correlated with its neighbours, a nugget far above the variance.  On both sides of each
rule, warp and CTA kernels, value and gradient, against the oracle.  Tolerances are the repository's (a term
within 1e-9 of max(|l_i|, 1), a gradient term within 1e-7 of the larger of itself and the mean, a
prediction within 1e-9); small predictions relative, to the 1e-8 of a small correlation."""
import numpy as np
import pytest
import torch

import oracle
from paper_2403_07412_gb300 import datagen
from tests import workloads as W

pytestmark = pytest.mark.gpu
SIZES = [37, 45, 50, 60, 63, 64, 90, 120]


@pytest.fixture(scope="module")
def V():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_07412_gb300 import build, vecchia

    build.build()
    oracle.build()
    return vecchia


def _check(V, m, theta, scale, n=None, order="random"):
    n = m + 250 if n is None else n
    xy = datagen.uniform_locations(n, datagen.BASE_SEED + 1030 + m)
    y = datagen.field_rff(xy, (1.0, 0.1, 0.5, 0.01), datagen.BASE_SEED + 1031, features=256)
    perm = oracle.order_random(n, datagen.BASE_SEED + 1032)
    y[perm] *= scale(n)  # by ordered position
    plan = V.Plan(xy, m, order=V.ORDER_GIVEN, perm=perm)
    yd = torch.as_tensor(y, device="cuda")
    want = oracle.vecchia_rows(xy[perm], y[perm], m, theta, want_grad=True)
    got = V.vecchia_loglik_terms(plan, yd, theta, want_grad=True).cpu().numpy()
    fwd = V.vecchia_loglik_terms(plan, yd, theta).cpu().numpy()
    lim = W.LOGLIK_RTOL * np.maximum(np.abs(want[:, 0]), 1.0)
    assert np.all(np.abs(fwd - want[:, 0]) <= lim)
    assert np.all(np.abs(got[:, 0] - want[:, 0]) <= lim)
    for k in (1, 2, 3):
        den = np.maximum(np.abs(want[:, k]), np.abs(want[:, k]).mean())
        assert np.all(np.abs(got[:, k] - want[:, k]) <= W.GRAD_RTOL * den), k


@pytest.mark.parametrize("m", SIZES)
def test_one_datum_far_above_the_others(V, m):
    _check(V, m, (1.0, 0.005, 0.5, 0.05), lambda n: np.where(np.arange(n) == 3, 1e9, 1.0))


@pytest.mark.parametrize("m", SIZES)
@pytest.mark.parametrize("period", [2, 3])  # every second or third datum: more or fewer than half are large
def test_some_data_above_the_others(V, m, period):
    _check(V, m, (1.0, 0.02, 1.5, 0.05), lambda n: np.where(np.arange(n) % period == 0, 1e3, 1.0))


@pytest.mark.parametrize("m", SIZES)
@pytest.mark.parametrize("beta", [3e-4, 2e-3, 5e-3, 1e-2])  # nearest neighbours' correlations from 1e-60 to 0.1
def test_weak_correlation(V, m, beta):
    _check(V, m, (1.3, beta, 0.5, 0.2), lambda n: 1.0)


@pytest.mark.parametrize("m", SIZES)
@pytest.mark.parametrize("tau2", [6.5e4, 6.6e4, 1e6])  # from 2^16 on
def test_large_nugget(V, m, tau2):
    n = m + 100
    xy = datagen.uniform_locations(n, datagen.BASE_SEED + 1040)
    y = np.sqrt(tau2) * datagen.rng(datagen.BASE_SEED + 1041).standard_normal(n)
    plan = V.Plan(xy, m, order=V.ORDER_GIVEN, perm=np.arange(n))
    yd, theta = torch.as_tensor(y, device="cuda"), (1.0, 0.1, 1.5, tau2)
    want = oracle.vecchia_rows(xy, y, m, theta, want_grad=True)
    got = V.vecchia_loglik_terms(plan, yd, theta, want_grad=True).cpu().numpy()
    lim = W.LOGLIK_RTOL * np.maximum(np.abs(want[:, 0]), 1.0)
    assert np.all(np.abs(got[:, 0] - want[:, 0]) <= lim)
    for k in (2, 3):
        den = np.maximum(np.abs(want[:, k]), np.abs(want[:, k]).mean())
        assert np.all(np.abs(got[:, k] - want[:, k]) <= W.GRAD_RTOL * den), k


@pytest.mark.parametrize("m", [5, 20, 37, 50, 60, 63])
@pytest.mark.parametrize("nu", [0.5, 1.5])
def test_prediction_far_from_all_data(V, m, nu):
    """Observed points in a cluster beside the origin, one far off so that the search grid spans the rest."""
    n, theta = 200, (1.2, 1.0, nu, 0.1)
    g = datagen.rng(datagen.BASE_SEED + 1050 + m)
    xy = np.concatenate([g.uniform(-0.5, 0.5, (n, 2)), [[1000.0, 0.0]]])
    y = 1.0 + 0.3 * g.standard_normal(n + 1)
    new = np.stack([np.array([0.7, 2.0, 5.0, 9.0, 20.0, 40.0, 60.0]), np.zeros(7)], 1)
    plan = V.Plan(xy, m, order=V.ORDER_RANDOM, seed=2)
    mean, var = V.vecchia_predict(plan, new, torch.as_tensor(y, device="cuda"), theta)
    wm, wv, _ = oracle.predict(xy, y, new, m, theta)
    mean, var = mean.cpu().numpy(), var.cpu().numpy()
    assert np.all(np.abs(wm[3:]) < 0.1) and np.abs(wm[-1]) < 1e-20
    assert np.all(np.abs(mean - wm) <= 1e-8 * np.abs(wm)), mean / wm - 1
    assert np.all(np.abs(var - wv) <= 1e-9)


@pytest.mark.parametrize("m", [50, 63, 64, 90])
def test_coincident_points_and_bad_data_there(V, m):
    n = m + 60
    xy = datagen.uniform_locations(n, datagen.BASE_SEED + 1060)
    y = datagen.rng(datagen.BASE_SEED + 1061).standard_normal(n)
    y[0] = 1e12  # in every early block
    xy[n - 1] = xy[n - 2]
    plan = V.Plan(xy, m, order=V.ORDER_GIVEN, perm=np.arange(n))
    for grad in (False, True):
        t = V.vecchia_loglik_terms(plan, torch.as_tensor(y, device="cuda"), (1.0, 1e-3, 0.5, 0.0), want_grad=grad).cpu().numpy()
        assert np.isnan(t[n - 1]).all() and np.isfinite(t[: n - 1]).all()
        assert plan.last_error() == (n - 1, V.ENOTPD)
    y[5] = np.nan
    touched = (plan.neighbors() == 5).any(1)
    touched[5] = True
    touched[n - 1] = True
    t = V.vecchia_loglik_terms(plan, torch.as_tensor(y, device="cuda"), (1.0, 0.1, 0.5, 0.0), want_grad=True).cpu().numpy()
    assert np.array_equal(np.isnan(t), np.repeat(touched[:, None], 4, 1))
    assert plan.last_error() == (5, V.EINVAL)
