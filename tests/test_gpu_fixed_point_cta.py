"""The CTA-per-location kernel's elimination in fixed point against the oracle: the edges of its
panels (a last panel of one to eight columns), every CTA size, as few locations as m allows, and the
corners of the scaling.  Tolerances are those of the full-warp blocks."""
import numpy as np
import pytest
import torch

from paper_2403_07412_gb300 import datagen
from tests import workloads as W
from tests.test_gpu_fixed_point import V, _check, _terms  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [64, 65, 70, 71, 72, 79, 80, 95, 96, 127, 128, 143, 150])
def test_panel_edges(V, m):  # noqa: F811
    _check(*_terms(V, m, (1.2, 0.08, 1.5, 0.02), n=m + 90))


@pytest.mark.parametrize("m", [64, 103, 150])
@pytest.mark.parametrize("threads", [64, 96, 128, 160, 192, 224, 256])
def test_cta_sizes(V, m, threads, monkeypatch):  # noqa: F811
    monkeypatch.setenv("VECCHIA_CTA_THREADS", str(threads))
    _check(*_terms(V, m, (1.2, 0.08, 0.5, 0.05), n=m + 1))


@pytest.mark.parametrize("theta", [(1.0, 0.1, 0.5, 0.0), (0.5, 0.05, 1.5, 8.0), (1e-3, 0.1, 0.5, 30.0), (1e6, 0.1, 1.0, 1e3)])
def test_scales(V, theta):  # noqa: F811
    _check(*_terms(V, 90, theta, n=300))


@pytest.mark.parametrize("yscale", [1e-120, 1e-9, 1e5, 1e120])
def test_data_far_from_sigma(V, yscale):  # noqa: F811
    got, fwd, want = _terms(V, 90, (1.0, 0.1, 0.5, 0.01), yscale=yscale, n=300)
    lim = W.LOGLIK_RTOL * np.maximum(np.abs(want[:, 0]), 1.0)
    assert np.all(np.abs(fwd - want[:, 0]) <= lim)
    assert np.all(np.abs(got[:, 0] - want[:, 0]) <= lim)


def test_failures(V):  # noqa: F811
    n = 300
    xy = datagen.uniform_locations(n, datagen.BASE_SEED + 970)
    y = datagen.field_rff(xy, (1.0, 0.1, 0.5, 0.01), 3, features=64)
    y[17] = np.inf
    plan = V.Plan(xy, 90, order=V.ORDER_RANDOM, seed=5)
    t = V.vecchia_loglik_terms(plan, torch.as_tensor(y, device="cuda"), (1.0, 0.1, 0.5, 0.01), want_grad=True).cpu().numpy()
    at = int(np.where(plan.perm() == 17)[0][0])
    touched = (plan.neighbors() == at).any(1)
    touched[at] = True
    assert np.array_equal(np.isnan(t), np.repeat(touched[:, None], 4, 1))
    assert plan.last_error() == (at, V.EINVAL)
    xy[1::7] = xy[0:-1:7][: len(xy[1::7])]  # without a nugget, blocks that hold a pair fail
    plan = V.Plan(xy, 90, order=V.ORDER_RANDOM, seed=7)
    yd = torch.as_tensor(datagen.rng(8).standard_normal(n), device="cuda")
    assert np.isnan(V.vecchia_loglik_terms(plan, yd, (1.0, 0.1, 0.5, 0.0)).cpu().numpy()).any()
    assert plan.last_error()[1] == V.ENOTPD
