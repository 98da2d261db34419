"""The full-warp blocks' elimination in fixed point against the oracle.

Larger blocks (m >= 37 forward, m >= 48 with the gradient) are eliminated in 64-bit fixed point
with the updates between panels of eight columns on the tensor cores.  The sizes are the
edges of panels and row slots (a last panel of one to eight columns, 38 to 65 rows); the
parameters are the corners of the scaling: no nugget, a nugget far above the variance, data far
above and far below sigma (the data row's units are chosen from both, and a block whose
residuals outgrow them is built again), duplicated points, a non-finite datum.  Tolerances are
the repository's: a term within 1e-9 of max(|l_i|, 1), a gradient term within 1e-7 of the larger of
itself and the mean.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2403_07412_gb300 import datagen
from tests import workloads as W

pytestmark = pytest.mark.gpu
N = 700


@pytest.fixture(scope="module")
def V():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_07412_gb300 import build, vecchia

    build.build()
    oracle.build()
    return vecchia


def _terms(V, m, theta, yscale=1.0, xy=None, n=N):
    xy = datagen.uniform_locations(n, datagen.BASE_SEED + 900 + m) if xy is None else xy
    n = len(xy)
    y = yscale * datagen.field_rff(xy, (1.0, 0.1, 0.5, 0.01), datagen.BASE_SEED + 901, features=256)
    perm = oracle.order_random(n, datagen.BASE_SEED + 902)
    plan = V.Plan(xy, m, order=V.ORDER_GIVEN, perm=perm)
    yd = torch.as_tensor(y, device="cuda")
    want = oracle.vecchia_rows(xy[perm], y[perm], m, theta, want_grad=True)
    got = V.vecchia_loglik_terms(plan, yd, theta, want_grad=True).cpu().numpy()
    fwd = V.vecchia_loglik_terms(plan, yd, theta).cpu().numpy()
    plan.close()
    return got, fwd, want


def _check(got, fwd, want):
    lim = W.LOGLIK_RTOL * np.maximum(np.abs(want[:, 0]), 1.0)
    assert np.all(np.abs(got[:, 0] - want[:, 0]) <= lim)
    assert np.all(np.abs(fwd - want[:, 0]) <= lim)
    for k in (1, 2, 3):
        den = np.maximum(np.abs(want[:, k]), np.abs(want[:, k]).mean())
        assert np.all(np.abs(got[:, k] - want[:, k]) <= W.GRAD_RTOL * den), k


@pytest.mark.parametrize("m", [37, 38, 39, 40, 46, 47, 48, 54, 55, 56, 61, 62, 63])
def test_panel_edges(V, m):
    _check(*_terms(V, m, (1.2, 0.08, 1.5, 0.02)))


@pytest.mark.parametrize("theta", [(1.0, 0.1, 0.5, 0.0), (1.3, 0.05, 1.5, 1.4), (0.5, 0.05, 1.5, 8.0), (1e-3, 0.1, 0.5, 30.0),
                                   (1e-6, 0.1, 0.5, 5.0), (1e-5, 0.1, 1.0, 1e-7), (1e6, 0.1, 1.0, 1e3)])
def test_scales(V, theta):
    _check(*_terms(V, 60, theta))


@pytest.mark.parametrize("yscale", [1e-120, 1e-9, 1e5, 1e120])
def test_data_far_from_sigma(V, yscale):
    got, fwd, want = _terms(V, 60, (1.0, 0.1, 0.5, 0.01), yscale=yscale)
    lim = W.LOGLIK_RTOL * np.maximum(np.abs(want[:, 0]), 1.0)
    assert np.all(np.abs(fwd - want[:, 0]) <= lim)
    assert np.all(np.abs(got[:, 0] - want[:, 0]) <= lim)


def test_duplicates(V):
    xy = datagen.uniform_locations(N, datagen.BASE_SEED + 950)
    xy[1::7] = xy[0:-1:7][: len(xy[1::7])]
    _check(*_terms(V, 60, (1.0, 0.1, 0.5, 0.05), xy=xy))  # a nugget keeps the blocks positive definite
    plan = V.Plan(xy, 60, order=V.ORDER_RANDOM, seed=7)  # without one, those that hold a pair fail
    yd = torch.as_tensor(datagen.rng(8).standard_normal(N), device="cuda")
    theta = (1.0, 0.1, 0.5, 0.0)
    got = V.vecchia_loglik_terms(plan, yd, theta, want_grad=True).cpu().numpy()
    fwd = V.vecchia_loglik_terms(plan, yd, theta).cpu().numpy()
    assert np.isnan(fwd).any() and np.array_equal(np.isnan(fwd), np.isnan(got[:, 0]))
    assert plan.last_error()[1] == V.ENOTPD


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_data(V, bad):
    xy = datagen.uniform_locations(N, datagen.BASE_SEED + 960)
    y = datagen.field_rff(xy, (1.0, 0.1, 0.5, 0.01), 3, features=64)
    y[17] = bad
    plan = V.Plan(xy, 60, order=V.ORDER_RANDOM, seed=5)
    yd = torch.as_tensor(y, device="cuda")
    t = V.vecchia_loglik_terms(plan, yd, (1.0, 0.1, 0.5, 0.01)).cpu().numpy()
    perm, nbr = plan.perm(), plan.neighbors()
    at = int(np.where(perm == 17)[0][0])
    touched = (nbr == at).any(1)
    touched[at] = True
    assert np.array_equal(np.isnan(t), touched)
    assert plan.last_error() == (at, V.EINVAL)
