"""A plan's first prediction on a stream that does not wait for the legacy default stream: the search grid it
lays out has to be in place before the kernel that reads it, on that stream and on any other that comes
next.  The grid's contents are exact, so conditioning sets are equal bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from paper_2403_07412_gb300 import datagen

pytestmark = pytest.mark.gpu
THETA = (1.2, 0.05, 1.5, 0.02)


@pytest.fixture(scope="module")
def V():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_07412_gb300 import build, vecchia

    build.build()
    oracle.build()
    return vecchia


@pytest.mark.parametrize("n", [60, 3000, 120_000])  # uploads below and above the size copied by staging alone
def test_first_prediction_on_side_streams(V, n):
    m = 10
    xy, new = datagen.uniform_locations(n, 31), datagen.uniform_locations(500, 32)
    y = torch.as_tensor(datagen.rng(33).standard_normal(n), device="cuda")
    want = oracle.predict(xy, y.cpu().numpy(), new, m, THETA)
    for _ in range(3):
        plan = V.Plan(xy, m, order=V.ORDER_RANDOM, seed=3)
        for _ in range(2):  # the first prediction, then one on another stream
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                mean, var, nbr = V.vecchia_predict(plan, new, y, THETA, return_neighbors=True)
                side.synchronize()
            np.testing.assert_array_equal(nbr, want[2])
            assert np.all(np.abs(mean.cpu().numpy() - want[0]) <= 1e-9 * np.maximum(np.abs(want[0]), 1.0))
            assert np.all(np.abs(var.cpu().numpy() - want[1]) <= 1e-9)
        plan.close()
