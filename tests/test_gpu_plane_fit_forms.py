"""Plane fitting with one pixel per thread (frames that do not fill the GPU) and with two
(larger frames): a small frame and the same frame as a corner of a larger one give the
same bits where the windows see the same depths."""
import pytest
import torch

import paper_2209_08241_gb300 as nrm
from test_gpu_strip import DEV, bits, depth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radius", [1, 2, 3, 4])
@pytest.mark.parametrize("dtype", ["f32", "u16"])
def test_small_frames_same_bits_as_large_ones(radius, dtype):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(radius)
    K = (300.0, 310.0, 80.3, 60.7)
    big = depth(640, 520, dtype, gen)
    for orient in (False, True):
        p = nrm.NormalParams(orient_to_camera=orient)
        n, m = nrm.NormalEstimator(K, 520, 640, p, dtype).plane_fit(big, radius)
        for W, H in [(160, 120), (161, 121), (33, 9), (31, 8), (32, 17), (608, 63), (1, 1), (2, 5), (65, 64)]:
            est = nrm.NormalEstimator(K, H, W, p, dtype)
            ns, ms = est.plane_fit(big[:H, :W].contiguous(), radius)
            est.sync_status()
            h, w = max(H - radius, 0), max(W - radius, 0)
            assert torch.equal(ms[:h, :w], m[:h, :w]), (W, H)
            assert torch.equal(bits(ns[:h, :w]), bits(n[:h, :w])), (W, H)
            assert int(ms[h:].sum()) == 0 and int(ms[:, w:].sum()) == 0
            assert not ns[h:].any() and not ns[:, w:].any()
