"""The adjoint around the edges of its tiles: frame sizes at and beside multiples of
every tile size, frames that TMA cannot load, distances of both kernel forms,
plain against batched (bit for bit) and, on small frames, against the
complex-step oracle with the tolerance of the adjoint (1e-3 relative)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2209_08241_gb300 as nrm

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def frame(H, W, pad, gen):
    d = torch.rand((H, W + pad), generator=gen, device=DEV) * 0.2 + 2.0
    d[torch.rand(d.shape, generator=gen, device=DEV) < 0.02] = 0.0
    return d[:, :W]


@pytest.mark.parametrize("alpha", [1, 2, 3, 4, 5])
def test_adjoint_tile_edges(alpha):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(alpha)
    b = nrm.BatchedEstimator(nrm.NormalParams(alpha=alpha))
    # (At alpha = 2 the last five take the walk, the others the gather.)
    for H, W, pad in [(23, 56, 0), (24, 57, 0), (25, 60, 4), (28, 61, 0), (29, 64, 0), (33, 120, 1), (57, 124, 0),
                      (28, 60, 0), (56, 120, 4), (84, 180, 0), (27, 59, 0), (55, 119, 1)]:
        K = (0.9 * W, 0.8 * W, 0.45 * W, 0.55 * H)
        d = frame(H, W, pad, gen)
        g = torch.randn((H, W + pad, 4), generator=gen, device=DEV)[:, :W]
        n = torch.empty((H, W + pad, 4), device=DEV)[:, :W]
        m = torch.empty((H, W + pad), dtype=torch.uint8, device=DEV)[:, :W]
        b([(d, K)], [(n, m)])
        out = torch.full((H, W + pad), 7.0, device=DEV)
        b.backward([(d, K)], [g], [m], [out[:, :W]])
        dc, gc, mc = d.contiguous(), g.contiguous(), m.contiguous()
        est = nrm.NormalEstimator(K, H, W, nrm.NormalParams(alpha=alpha))
        one = est.backward(dc, gc, mc)
        assert torch.equal(one, out[:, :W].contiguous()), (alpha, H, W)
        assert bool((out[:, W:] == 7.0).all())
        ref = oracle.vjp(dc.cpu().numpy(), K, gc[..., :3].double().cpu().numpy(), mc.cpu().numpy(), alpha=alpha,
                         crop=(0, 0, H, W))
        got = one.double().cpu().numpy()
        big = np.abs(ref) > 1e-3 * np.abs(ref).max()
        assert (np.abs(got - ref)[big] <= 1e-3 * np.abs(ref)[big]).all(), (alpha, H, W)
        est.sync_status()
    b.sync_status()
