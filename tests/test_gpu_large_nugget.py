"""A nugget many orders above the variance: value and the gradient in tau2 of blocks eliminated in fixed
point (the first ones padded) against the oracle, to the repository's tolerances.  The gradient in beta
vanishes with sigma2 / tau2 and has to be finite and as small; that in sigma2 is a difference of terms
sigma2 / tau2 times larger, which FP64 does not resolve, and has to be finite."""
import numpy as np
import pytest

from tests import workloads as W
from tests.test_gpu_fixed_point import V, _terms  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [60, 90])
@pytest.mark.parametrize("ratio", [1e9, 1e18, 1e20, 1e25, 1e40])
def test_large_nugget(V, m, ratio):  # noqa: F811
    got, fwd, want = _terms(V, m, (1.0, 0.1, 0.5, ratio), n=200)
    lim = W.LOGLIK_RTOL * np.maximum(np.abs(want[:, 0]), 1.0)
    assert np.all(np.abs(got[:, 0] - want[:, 0]) <= lim) and np.all(np.abs(fwd - want[:, 0]) <= lim)
    den = np.maximum(np.abs(want[:, 3]), np.abs(want[:, 3]).mean())
    assert np.all(np.abs(got[:, 3] - want[:, 3]) <= W.GRAD_RTOL * den)
    assert np.all(np.isfinite(got)) and np.all(np.abs(got[:, 2]) <= 100.0 * m * m / ratio)
