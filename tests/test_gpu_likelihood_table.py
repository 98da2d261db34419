"""The likelihood kernels' covariance table over smoothness and distance, through the terms of small
blocks, against the oracle: the smallest and large nu, integers and beside them, distances from below the
table's first interval to beyond its last.  Tolerances are the repository's for terms (the fixed-point
table is closer to rho than the earlier one they were set for)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2403_07412_gb300 import datagen
from tests import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu", [0.1, 0.5, 0.9999, 1.0, 1.0001, 2.0, 3.7, 10.0, 40.0])
@pytest.mark.parametrize("beta", [1e-4, 0.05, 3.0])
def test_terms_over_nu_and_distance(nu, beta):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_07412_gb300 import build, vecchia as V

    build.build()
    oracle.build()
    n, m, theta = 160, 7, (1.3, beta, nu, 0.4)
    xy = datagen.uniform_locations(n, 41)
    xy[1::5] = xy[0:-1:5][: len(xy[1::5])] + 1e-7  # pairs far closer than the table's first interval
    y = datagen.rng(42).standard_normal(n)
    perm = oracle.order_random(n, 43)
    plan = V.Plan(xy, m, order=V.ORDER_GIVEN, perm=perm)
    try:
        want = oracle.vecchia_rows(xy[perm], y[perm], m, theta, want_grad=True)
    except oracle.OracleNotPD:  # its x^nu K_nu(x) is 0 times infinity at nu = 40, x = 3e-8
        assert nu == 40.0 and beta == 3.0
        pytest.skip("outside the oracle's range")
    got = V.vecchia_loglik_terms(plan, torch.as_tensor(y, device="cuda"), theta, want_grad=True).cpu().numpy()
    assert np.all(np.abs(got[:, 0] - want[:, 0]) <= W.LOGLIK_RTOL * np.maximum(np.abs(want[:, 0]), 1.0))
    for k in (1, 2, 3):
        den = np.maximum(np.abs(want[:, k]), np.abs(want[:, k]).mean())
        assert np.all(np.abs(got[:, k] - want[:, k]) <= W.GRAD_RTOL * den), k
