"""The adjoint at the distances above 5, up to the largest one that the library takes:
single and batched entry points (parameter block and descriptor ring) give the
same bits, and crops match the complex-step oracle with the tolerance of the
adjoint (1e-3 relative)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2209_08241_gb300 as nrm

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("alpha", [6, 8, 15, 16])
def test_adjoint_at_large_distances(alpha):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(alpha)
    b = nrm.BatchedEstimator(nrm.NormalParams(alpha=alpha))
    items, grads, masks = [], [], []
    for H, W in [(33, 65), (32, 64), (97, 131), (160, 128), (1, 40)]:
        K = (0.9 * W, 0.8 * W, 0.45 * W, 0.55 * H)
        d = torch.rand((H, W), generator=gen, device=DEV) * 0.2 + 2.0
        d[torch.rand((H, W), generator=gen, device=DEV) < 0.01] = 0.0
        (n, m), = b([(d, K)])
        items.append((d, K))
        grads.append(torch.randn((H, W, 4), generator=gen, device=DEV))
        masks.append(m)
        est = nrm.NormalEstimator(K, H, W, nrm.NormalParams(alpha=alpha))
        one = est.backward(d, grads[-1], m)
        est.sync_status()
        ref = oracle.vjp(d.cpu().numpy(), K, grads[-1][..., :3].double().cpu().numpy(), m.cpu().numpy(), alpha=alpha,
                         crop=(0, 0, H, W))
        big = np.abs(ref) > 1e-3 * np.abs(ref).max()
        got = one.double().cpu().numpy()
        assert (np.abs(got - ref)[big] <= 1e-3 * np.abs(ref)[big]).all(), (alpha, H, W)
        assert np.abs(got - ref)[~big].max(initial=0.0) <= 1e-3 * np.abs(ref).max(initial=0.0)
    for times in (1, 13):
        for got, (d, K), g, m in zip(b.backward(items * times, grads * times, masks * times), items, grads, masks):
            est = nrm.NormalEstimator(K, *d.shape, nrm.NormalParams(alpha=alpha))
            assert torch.equal(got, est.backward(d, g, m)), (alpha, times, d.shape)
    b.sync_status()
