"""nrm_cosine_loss_scale on masks of few, long rows with gaps behind them, where a row is
counted in several parts: exact counts around the parts' lengths, at every
alignment."""
import pytest
import torch

import paper_2209_08241_gb300 as nrm

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("W", [511, 512, 513, 1025, 8191, 131072, 131089, 300007])
@pytest.mark.parametrize("H", [1, 2, 7, 129, 257])
def test_counts_of_long_rows(H, W):
    if H > 7 and W > 10000:
        W //= 16
    gen = torch.Generator(device=DEV)
    gen.manual_seed(H * 1000 + W)
    b = nrm.BatchedEstimator()
    items, grads, masks = [], [], []
    for i in range(4):
        pad = (1, 16, 31, 5)[i]
        buf = torch.randint(0, 256, (5 * i + H * (W + pad),), generator=gen, device=DEV).to(torch.uint8)
        buf[torch.rand(buf.shape, generator=gen, device=DEV) < 0.4] = 0
        masks.append(buf[5 * i:].view(H, W + pad)[:, :W])
        grads.append(torch.zeros((H, W + pad, 4), device=DEV)[:, :W])
        items.append((torch.ones((H, W), device=DEV), (100.0, 100.0, 1.0, 1.0)))
    arr, _ = b.make_grad_frames(items, grads, masks)
    for _ in range(2):
        got = b.cosine_loss_scale(arr, len(items))
        for i, m in enumerate(masks):
            n = int((m != 0).sum())
            assert float(got[i]) == float(torch.tensor(-1.0) / torch.tensor(float(max(n, 1)))), (i, n)
