"""A plan's first prediction and a batch's first call on streams that do not wait for the legacy default
stream: what those calls lay out on the device once has to be in place before the kernels that read it, on
that stream and on any other that comes next.  The search grid's and the layout's contents are exact, so
conditioning sets are equal bit for bit and results equal those of a later call."""
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


def test_first_batched_call_on_a_side_stream(V):
    sizes = [(700, 10), (400, 30), (300, 60)]
    V.vecchia_batched_prepare([0.5, 1.5])
    thetas = torch.as_tensor(np.tile([THETA, (0.8, 0.1, 0.5, 0.1)], (3, 1, 1)), device="cuda").contiguous()
    plans = [V.Plan(datagen.uniform_locations(n, 40 + m), m, order=V.ORDER_RANDOM, seed=4) for n, m in sizes]
    ys = [torch.as_tensor(datagen.rng(50 + m).standard_normal(n), device="cuda") for n, m in sizes]
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        batch = V.Batch(plans, ys, 2, want_grad=True)
        first = batch.run(thetas).clone()
        side.synchronize()
    again = batch.run(thetas).cpu().numpy()
    assert np.array_equal(first.cpu().numpy(), again) and np.isfinite(again).all()
