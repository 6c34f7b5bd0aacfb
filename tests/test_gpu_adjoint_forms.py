"""Both forms of the adjoint around the edges of their tiles, at the distances that have
two: frames that TMA loads and frames of odd pitches, single and batched (bit for bit
the same), against the complex-step oracle with the tolerance of the adjoint (1e-3
relative). Which form a frame takes is checked on the host side alone, so that
neither can drop out of this test unseen."""
import numpy as np
import pytest
import torch

import fake_gpu
import oracle
import paper_2209_08241_gb300 as nrm
from test_gpu_adjoint_tiles import DEV, frame

GATHER = [(31, 63), (32, 64), (29, 65), (64, 127), (63, 128), (32, 129), (64, 61)]  # (H, W) at alpha 2
WALK = [(28, 60), (56, 120), (33, 65), (65, 129), (84, 180), (28, 65), (33, 60)]


@pytest.mark.parametrize("alpha,sizes,form", [(2, GATHER, "walk=0"), (2, WALK, "walk=1"), (1, WALK, "walk=0"),
                                              (3, GATHER, "walk=1"), (4, GATHER, "walk=1")])
def test_forms(alpha, sizes, form):
    lib = fake_gpu.load()
    B = fake_gpu.BASE
    for H, W in sizes:
        lib.fake_reset()
        h = fake_gpu.handle(lib, H, W, alpha=alpha)
        assert lib.nrm_backward(h, B, B, B, B, None) == 0
        assert lib.nrm_backward_batched(h, fake_gpu.grad_frames([(W, H)]), 1, None) == 0
        assert all(form in ln for ln in fake_gpu.log(lib)) and len(fake_gpu.log(lib)) == 2, (alpha, H, W)
        lib.nrm_destroy(h)
    lib.fake_reset()


@pytest.mark.gpu
@pytest.mark.parametrize("alpha,sizes", [(2, GATHER), (2, WALK), (3, GATHER), (4, GATHER), (1, WALK)])
@pytest.mark.parametrize("pad", [0, 1, 4])
def test_tile_edges_of_either_form(alpha, sizes, pad):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(alpha + 10 * pad)
    b = nrm.BatchedEstimator(nrm.NormalParams(alpha=alpha))
    for H, W in sizes:
        K = (0.9 * W, 0.8 * W, 0.45 * W, 0.55 * H)
        d = frame(H, W, pad, gen)
        g = torch.randn((H, W + pad, 4), generator=gen, device=DEV)[:, :W]
        n = torch.empty((H, W + pad, 4), device=DEV)[:, :W]
        m = torch.empty((H, W + pad), dtype=torch.uint8, device=DEV)[:, :W]
        b([(d, K)], [(n, m)])
        out = torch.full((H, W + pad), 7.0, device=DEV)
        b.backward([(d, K)], [g], [m], [out[:, :W]])
        assert bool((out[:, W:] == 7.0).all())
        dc, gc, mc = d.contiguous(), g.contiguous(), m.contiguous()
        est = nrm.NormalEstimator(K, H, W, nrm.NormalParams(alpha=alpha))
        one = est.backward(dc, gc, mc)
        assert torch.equal(one, out[:, :W].contiguous()), (alpha, H, W)
        est.sync_status()
        ref = oracle.vjp(dc.cpu().numpy(), K, gc[..., :3].double().cpu().numpy(), mc.cpu().numpy(), alpha=alpha,
                         crop=(0, 0, H, W))
        big = np.abs(ref) > 1e-3 * np.abs(ref).max()
        got = one.double().cpu().numpy()
        assert (np.abs(got - ref)[big] <= 1e-3 * np.abs(ref)[big]).all(), (alpha, H, W)
    b.sync_status()
