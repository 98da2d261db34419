"""Calls of different block sizes in any order: a size's launch shape is searched once, which tries the kernels' shared
memory limits, and later calls of sizes found before have to set theirs again.  Results equal the first ones
bit for bit."""
import itertools

import numpy as np
import pytest
import torch

from paper_2403_07412_gb300 import datagen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", list(itertools.permutations((40, 50, 60), 3)) + [(50, 53, 63, 37), (63, 37, 52, 54), (45, 120, 64, 45)])
def test_sizes_in_turn(sizes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_07412_gb300 import build, vecchia as V

    build.build()
    n, theta = 3000, (1.0, 0.1, 1.5, 0.05)
    xy = datagen.uniform_locations(n, 81)
    y = torch.as_tensor(datagen.rng(82).standard_normal(n), device="cuda")
    plans = [V.Plan(xy, m, order=V.ORDER_MORTON) for m in sizes]
    first = {}
    for k in (0, 1, 0, 2, 1, 0, *range(len(sizes)), *reversed(range(len(sizes)))):
        got = (V.vecchia_loglik(plans[k], y, theta).cpu().numpy(), V.vecchia_loglik_grad(plans[k], y, theta).cpu().numpy(),
               V.vecchia_loglik_range(plans[k], y, theta, 100, 2100).cpu().numpy())
        assert all(np.isfinite(g).all() for g in got)
        for a, b in zip(first.setdefault(k, got), got):
            assert np.array_equal(a, b)
