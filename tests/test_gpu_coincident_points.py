"""Blocks that hold two coincident points and no nugget: singular, so every one of them has to be reported as
not positive definite, and no other.  An elimination in fixed point leaves such a pivot at some units of its
own rounding, of either sign; the sizes are those where the last panel holds the location alone (m a multiple
of 8) and others, of the full-warp and the CTA kernels."""
import numpy as np
import pytest
import torch

from paper_2403_07412_gb300 import datagen

pytestmark = pytest.mark.gpu
THETA = (1.0, 0.1, 0.5, 0.0)


@pytest.fixture(scope="module")
def V():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_07412_gb300 import build, vecchia

    build.build()
    return vecchia


def _case(V, m, near, seed):
    """n locations in the given order; the later point of each pair comes `near` or `far` after the earlier."""
    n = m + 160
    g = datagen.rng(seed)
    xy = datagen.uniform_locations(n, seed)
    later = np.arange(m + 20, n, 7) if near else np.arange(9, n, 31)
    for i in later:
        xy[i] = xy[g.integers(0, i)]
    plan = V.Plan(xy, m, order=V.ORDER_GIVEN, perm=np.arange(n))
    nbr = plan.neighbors()
    own, pair = np.zeros(n, bool), np.zeros(n, bool)
    for i in range(n):
        j = xy[nbr[i][nbr[i] >= 0]]
        own[i] = len(j) > 0 and (j == xy[i]).all(1).any()
        pair[i] = len(np.unique(j, axis=0)) < len(j)
    return plan, torch.as_tensor(g.standard_normal(n), device="cuda"), own, pair


@pytest.mark.parametrize("m", [37, 40, 48, 56, 60, 63, 64, 72, 90, 120, 144, 150])
@pytest.mark.parametrize("near", [True, False])
def test_every_singular_block_is_reported(V, m, near):
    plan, y, own, pair = _case(V, m, near, datagen.BASE_SEED + 980 + m)
    bad = own | pair
    fwd = V.vecchia_loglik_terms(plan, y, THETA).cpu().numpy()
    assert np.array_equal(np.isnan(fwd), bad)
    assert plan.last_error() == (int(np.flatnonzero(bad)[0]), V.ENOTPD)
    got = V.vecchia_loglik_terms(plan, y, THETA, want_grad=True).cpu().numpy()
    if m >= 50:  # smaller blocks take the gradient in FP64, whose pivot at a pair of neighbours may round upwards
        assert np.array_equal(np.isnan(got), np.repeat(bad[:, None], 4, 1))
    assert np.isnan(got[own]).all() and not np.isnan(got[~bad]).any()


@pytest.mark.parametrize("m", [40, 60, 120])
def test_the_smallest_nugget_keeps_them(V, m):
    """With tau2 = 2^-40 sigma2 the same blocks are positive definite by far more than any rounding."""
    plan, y, own, pair = _case(V, m, True, datagen.BASE_SEED + 990 + m)
    t = V.vecchia_loglik_terms(plan, y, (1.0, 0.1, 0.5, 2.0**-40), want_grad=True).cpu().numpy()
    assert (own | pair).any() and np.isfinite(t).all()
