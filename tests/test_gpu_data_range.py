"""Data of very different sizes in one block against the oracle: a wild value among its neighbours, a field
whose amplitude changes across the domain, mostly zeros.  A datum must not cost its neighbours their digits.
Tolerances are the repository's (a term within 1e-9 of max(|l_i|, 1), a gradient term within 1e-7 of the
larger of itself and the mean)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2403_07412_gb300 import datagen
from tests import workloads as W

pytestmark = pytest.mark.gpu
SIZES = [10, 30, 40, 45, 60, 63, 64, 90, 120]


@pytest.fixture(scope="module")
def V():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_07412_gb300 import build, vecchia

    build.build()
    oracle.build()
    return vecchia


def _check(V, m, theta, scale):
    n = m + 300
    xy = datagen.uniform_locations(n, datagen.BASE_SEED + 1000 + m)
    y = datagen.field_rff(xy, (1.0, 0.1, 0.5, 0.01), datagen.BASE_SEED + 1001, features=256) * scale(xy, n)
    perm = oracle.order_random(n, datagen.BASE_SEED + 1002)
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
@pytest.mark.parametrize("factor", [1e4, 1e7])
def test_one_wild_datum(V, m, factor):
    _check(V, m, (1.0, 0.005, 0.5, 0.05), lambda xy, n: np.where(np.arange(n) == 17, factor, 1.0))


@pytest.mark.parametrize("m", SIZES)
def test_amplitude_over_the_domain(V, m):
    _check(V, m, (1.0, 0.01, 1.5, 0.05), lambda xy, n: 10.0 ** (6.0 * xy[:, 0] - 3.0))


@pytest.mark.parametrize("m", SIZES)
def test_mostly_zeros(V, m):
    _check(V, m, (1.0, 0.05, 1.5, 0.05), lambda xy, n: (np.arange(n) % 5 == 0) * 1.0)


@pytest.mark.parametrize("m", [40, 60, 63, 64, 120])
@pytest.mark.parametrize("theta", [(0.3, 0.1, 1.5, 0.003), (1.0, 0.3, 1.0, 1e-4), (1e-8, 0.1, 1.5, 1e-10)])
def test_rough_data_under_a_smooth_covariance(V, m, theta):
    """White noise where the covariance expects a smooth field: the whitened data are far above sigma."""
    n = m + 300
    xy = datagen.uniform_locations(n, datagen.BASE_SEED + 1010 + m)
    y = datagen.rng(datagen.BASE_SEED + 1011).standard_normal(n)
    perm = oracle.order_random(n, datagen.BASE_SEED + 1012)
    plan = V.Plan(xy, m, order=V.ORDER_GIVEN, perm=perm)
    want = oracle.vecchia_rows(xy[perm], y[perm], m, theta)
    fwd = V.vecchia_loglik_terms(plan, torch.as_tensor(y, device="cuda"), theta).cpu().numpy()
    assert np.all(np.abs(fwd - want) <= W.LOGLIK_RTOL * np.maximum(np.abs(want), 1.0))
