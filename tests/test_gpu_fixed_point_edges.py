"""Edges of the fixed-point sizes that the other tests pass by: the gradient's first size (m = 50) and a last panel
of every width for the warp and the CTA kernel, the gradient of data far from sigma, and the sphere with both
eliminations.  Against the oracle, to the repository's tolerances (a term within 1e-9 of max(|l_i|, 1), a
gradient term within 1e-7 of the larger of itself and the mean)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2403_07412_gb300 import datagen
from tests import workloads as W
from tests.test_gpu_fixed_point import V, _check, _terms  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [41, 42, 43, 44, 45, 49, 50, 51, 52, 53, 57, 58, 59, 60])
def test_warp_panel_widths(V, m):  # noqa: F811
    _check(*_terms(V, m, (1.2, 0.08, 1.5, 0.02), n=300))


@pytest.mark.parametrize("m", [66, 67, 68, 69, 74, 75, 76, 77, 78, 141, 142, 149])
def test_cta_panel_widths(V, m):  # noqa: F811
    _check(*_terms(V, m, (1.2, 0.08, 1.5, 0.02), n=m + 60))


@pytest.mark.parametrize("m", [60, 90])
@pytest.mark.parametrize("yscale", [1e-9, 1e5])
def test_gradient_of_data_far_from_sigma(V, m, yscale):  # noqa: F811
    _check(*_terms(V, m, (1.0, 0.1, 0.5, 0.01), yscale=yscale, n=300))


@pytest.mark.parametrize("m", [40, 55, 63, 90])
@pytest.mark.parametrize("beta", [2.0, 60.0, 800.0])  # km: neighbours some 400 km apart, from hardly correlated to strongly
@pytest.mark.parametrize("wild", [1.0, 1e4])
def test_sphere(V, m, beta, wild):  # noqa: F811
    n, radius, theta = m + 200, 6371.0, (1.2, beta, 0.8, 0.1)
    lonlat = datagen.sphere_locations(n, datagen.BASE_SEED + 1070)
    y = datagen.rng(datagen.BASE_SEED + 1071).standard_normal(n)
    perm = oracle.order_random(n, 5)
    y[perm[11]] *= wild
    plan = V.Plan(lonlat, m, order=V.ORDER_GIVEN, perm=perm, radius=radius)
    plan.set_kernel(V.KERNEL_POWEXP)
    yd = torch.as_tensor(y, device="cuda")
    want = oracle.vecchia_rows(lonlat[perm], y[perm], m, theta, want_grad=True, family=1, radius=radius)
    got = V.vecchia_loglik_terms(plan, yd, theta, want_grad=True).cpu().numpy()
    fwd = V.vecchia_loglik_terms(plan, yd, theta).cpu().numpy()
    lim = W.LOGLIK_RTOL * np.maximum(np.abs(want[:, 0]), 1.0)
    assert np.all(np.abs(fwd - want[:, 0]) <= lim) and np.all(np.abs(got[:, 0] - want[:, 0]) <= lim)
    for k in (1, 2, 3):
        den = np.maximum(np.abs(want[:, k]), np.abs(want[:, k]).mean())
        assert np.all(np.abs(got[:, k] - want[:, k]) <= W.GRAD_RTOL * den), k
