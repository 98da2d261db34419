"""The batched call's scratch stays bounded however large the batch: one 32-byte record an item, some 64 items for
each resident warp of a class (16 warps an SM at most), and one at least for each (field, theta)."""
import numpy as np
import pytest
import torch

from paper_2403_07412_gb300 import datagen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,ntheta", [(200_000, 4, 300), (100_000, 20, 200)])
def test_records_of_a_large_batch(n, m, ntheta):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_07412_gb300 import build, vecchia as V

    build.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    V.vecchia_batched_prepare([0.5])
    plan = V.Plan(datagen.uniform_locations(n, 71), m, order=V.ORDER_MORTON)
    y = torch.as_tensor(datagen.rng(72).standard_normal(n), device="cuda")
    g = datagen.rng(73)
    th = np.stack([g.uniform(0.5, 2.0, ntheta), g.uniform(0.02, 0.1, ntheta), np.full(ntheta, 0.5), g.uniform(0.01, 0.1, ntheta)], 1)
    thetas = torch.as_tensor(th[None], device="cuda").contiguous()
    out = torch.empty((1, ntheta, 4), dtype=torch.float64, device="cuda")
    small = V.Batch([plan], [y], 1, want_grad=True)  # loads the kernels
    small.run(thetas[:, :1].contiguous())
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    V.Batch([plan], [y], ntheta, want_grad=True).run(thetas, out)
    torch.cuda.synchronize()
    grown = before - torch.cuda.mem_get_info()[0]
    assert grown <= 1.2 * 32 * (64 * 16 * sms + ntheta) + 3 * 2**21  # and three allocations' granularity
    got = out.cpu().numpy()[0]
    for t in (0, ntheta // 2, ntheta - 1):  # against the single-field call: the same terms, other order of the additions
        one = V.vecchia_loglik_grad(plan, y, th[t]).cpu().numpy()
        assert np.all(np.abs(got[t] - one) <= 1e-9 * np.maximum(np.abs(one), n))
