"""Batches whose fields run as several kernel classes, with items of one to eight steps: the sizes
at the edges of the lanes-per-location classes, one location more than an item holds, few and many."""
import numpy as np
import pytest
import torch

from paper_2403_07412_gb300 import datagen
from tests import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,ms", [
    ((61, 62, 200, 65), (60, 60, 48, 47)),          # as few locations as m allows; FP64 and fixed point
    ((17, 400, 33, 9), (15, 16, 31, 7)),            # narrow groups
    ((20_001, 301, 9_999, 5_003), (10, 63, 25, 36)),  # one class with eight-step items, others with one
    ((4_097,), (1,)),
])
@pytest.mark.parametrize("grad", [True, False])
def test_batch_of_classes_matches_single_field_calls(sizes, ms, grad):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_07412_gb300 import vecchia as V

    V.vecchia_batched_prepare([0.5, 1.0, 1.5])
    plans, ys = [], []
    for f, (n, m) in enumerate(zip(sizes, ms)):
        xy = datagen.uniform_locations(n, 50 + f)
        plans.append(V.Plan(xy, m, order=V.ORDER_RANDOM, seed=60 + f))
        ys.append(torch.as_tensor(datagen.field_rff(xy, (1.0, 0.05, 1.0, 0.02), 70 + f, features=128), device="cuda"))
    nth = 3
    thetas = datagen.theta_candidates(len(sizes), nth, 7)
    td = torch.as_tensor(thetas, device="cuda").contiguous()
    b = V.Batch(plans, ys, nth, want_grad=grad)
    first = b.run(td).cpu().numpy()
    # another layout of the same kernels in between, then the first one again
    V.Batch(plans[:1], ys[:1], 1, want_grad=grad).run(td[:1, :1].contiguous())
    out = b.run(td).cpu().numpy()
    np.testing.assert_array_equal(first, out)
    for f in range(len(sizes)):
        for t in range(nth):
            terms = V.vecchia_loglik_terms(plans[f], ys[f], thetas[f, t], want_grad=True).cpu().numpy()
            want, den = terms.sum(0), np.abs(terms).sum(0)
            assert abs(out[f, t, 0] - want[0]) <= W.LOGLIK_RTOL * den[0], (f, t)
            for k in (1, 2, 3) if grad else ():
                assert abs(out[f, t, k] - want[k]) <= W.GRAD_RTOL * den[k], (f, t, k)
