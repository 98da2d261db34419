"""Blocks whose factor's rows are nearly constant: locations that almost coincide, under a nugget from the size of
the variance to far above it.  The digits of such rows do not spread over their range but repeat from column to
column, which makes the digit sums of the tensor-core updates as large as they get.  Value and the gradient in
tau2 against the oracle, to the repository's tolerances; the others (differences of terms sigma2 / tau2 times
larger) have to be finite."""
import numpy as np
import pytest
import torch

import oracle
from paper_2403_07412_gb300 import datagen
from tests import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [60, 63, 64, 120, 150])
@pytest.mark.parametrize("ratio", [0.5, 30.0, 1e3, 6e4, 1e6, 1e9, 1e10])
def test_near_coincident_locations(m, ratio):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_07412_gb300 import build, vecchia as V

    build.build()
    oracle.build()
    n, theta = m + 60, (1.0, 0.3, 1.5, ratio)
    g = datagen.rng(datagen.BASE_SEED + 1020 + m)
    xy = 0.5 + 1e-7 * datagen.uniform_locations(n, datagen.BASE_SEED + 1021)
    y = np.sqrt(ratio) * g.standard_normal(n) + g.standard_normal()
    plan = V.Plan(xy, m, order=V.ORDER_GIVEN, perm=np.arange(n))
    yd = torch.as_tensor(y, device="cuda")
    want = oracle.vecchia_rows(xy, y, m, theta, want_grad=True)
    got = V.vecchia_loglik_terms(plan, yd, theta, want_grad=True).cpu().numpy()
    fwd = V.vecchia_loglik_terms(plan, yd, theta).cpu().numpy()
    lim = W.LOGLIK_RTOL * np.maximum(np.abs(want[:, 0]), 1.0)
    assert np.all(np.abs(got[:, 0] - want[:, 0]) <= lim) and np.all(np.abs(fwd - want[:, 0]) <= lim)
    den = np.maximum(np.abs(want[:, 3]), np.abs(want[:, 3]).mean())
    assert np.all(np.abs(got[:, 3] - want[:, 3]) <= W.GRAD_RTOL * den)
    assert np.isfinite(got).all()
