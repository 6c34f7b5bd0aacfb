"""nrm_cosine_loss_scale at every alignment and pitch of the masks, for byte
values other than 1, against exact counts."""
import pytest
import torch

import paper_2209_08241_gb300 as nrm

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("W", [1, 15, 16, 17, 33, 512, 641])
@pytest.mark.parametrize("H", [1, 3, 300])
def test_loss_scale_counts(H, W):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(H * 1000 + W)
    b = nrm.BatchedEstimator()
    items, grads, masks = [], [], []
    for i in range(17):
        pad = (0, 0, 1, 16, 31)[i % 5]
        buf = torch.randint(0, 256, (i + H * (W + pad),), generator=gen, device=DEV).to(torch.uint8)
        buf[torch.rand(buf.shape, generator=gen, device=DEV) < 0.4] = 0
        masks.append(buf[i:].view(H, W + pad)[:, :W])
        grads.append(torch.zeros((H, W + pad, 4), device=DEV)[:, :W])
        items.append((torch.ones((H, W), device=DEV), (100.0, 100.0, 1.0, 1.0)))
    arr, _ = b.make_grad_frames(items, grads, masks)
    got = b.cosine_loss_scale(arr, len(items))
    for i, m in enumerate(masks):
        n = int((m != 0).sum())
        assert float(got[i]) == float(torch.tensor(-1.0) / torch.tensor(float(max(n, 1)))), (i, n)
