"""The angle MSE around the edges of its work split: rows of one pixel up to
several pieces of 128, pitched maps, more pieces than the grid has warps (several
flushes to FP64), and stale shared memory behind a ragged piece. Against the
FP64 oracle with the tolerance of the sums (1e-4 relative, exact counts)."""
import pytest
import torch

import paper_2209_08241_gb300 as nrm
from oracle import evaluation

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def maps(H, W, pitch, gen):
    n = torch.randn((H, pitch, 4), generator=gen, device=DEV)
    n[..., 0] += 3.0  # phi away from its 0 / 2 pi cut
    n[..., 0].abs_().add_(0.5)
    n[..., 1].abs_().add_(0.5)
    n[..., 3] = 0.0
    n = n / n.norm(dim=-1, keepdim=True)
    v = (torch.rand((H, pitch), generator=gen, device=DEV) < 0.8).to(torch.uint8)
    return n[:, :W], v[:, :W]


@pytest.mark.parametrize("H,W,pad", [(1, 1, 0), (3, 127, 0), (5, 128, 3), (40, 129, 0), (33, 257, 1), (2, 4095, 0),
                                     (1200, 3000, 8)])
def test_angle_mse_pieces(H, W, pad):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(H * 7 + W)
    est = nrm.NormalEstimator((100.0, 100.0, 1.0, 1.0), 8, 8)
    nan = torch.full((512, 4096, 4), float("nan"), device=DEV)
    on = torch.ones((512, 4096), dtype=torch.uint8, device=DEV)
    nrm.angle_mse(est, nan, on, nan, on)  # leaves NaN in every SM's shared memory
    na, va = maps(H, W, W + pad, gen)
    nb, vb = maps(H, W, W + pad, gen)
    out = nrm.angle_mse(est, na, va, nb, vb)
    assert torch.equal(out, nrm.angle_mse(est, na, va, nb, vb))
    mt, mp, cnt = evaluation.angle_mse(na.double().cpu().numpy(), va.cpu().numpy(), nb.double().cpu().numpy(),
                                       vb.cpu().numpy())
    got = out.cpu().numpy()
    assert int(got[2]) == cnt
    if cnt:
        assert got[0] == pytest.approx(mt, rel=1e-4)
        assert got[1] == pytest.approx(mp, rel=1e-4)
    est.sync_status()
