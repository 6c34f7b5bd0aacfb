"""The batched multi-scale kernels against each other, on batches that reach the strip
kernel (tests/test_multiscale_routes.py checks on the CPU that these do): each
frame bit for bit equal to the run-time-distance kernel on the same frame with
an odd output pitch, outputs in buffers with gaps that must keep their contents."""
import pytest
import torch

import paper_2209_08241_gb300 as nrm
from test_gpu_strip import DEV, assert_same, depth
from test_gpu_strip_routes import OUT, Buffers, bits, cameras

pytestmark = pytest.mark.gpu
SIZES = [(4, 1), (8, 5), (124, 63), (128, 64), (136, 65), (256, 7), (264, 129), (1032, 97), (1920, 1281)]
SMALL = [(64, 48), (128, 64), (136, 65), (320, 240)]


@pytest.mark.parametrize("form", ["pair", "quad"])
@pytest.mark.parametrize("K", [2, 3, 4, 5, 6])
@pytest.mark.parametrize("out", OUT)
def test_same_bits(form, K, out):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(K)
    items = [(depth(W, H, t, gen), cameras(W, H)) for W, H in SIZES for t in ("f32", "u16")
             if W * (2 if t == "u16" else 4) % 16 == 0]
    for mask, tau, sign in (("secant", 12.0, False), ("raw", 1e-3, True)):
        b = nrm.BatchedEstimator(nrm.NormalParams(out_dtype=out, mask_mode=mask, tau=tau, orient_to_camera=sign))
        got = []
        for gaps in ([(8 * (i % 2), 8) for i in range(len(items))], [(1, 3)] * len(items)):
            buf = Buffers(items, out, gaps)
            b.multiscale(items, range(1, K + 1), form, outputs=buf.views)
            got.append([(bits(n).clone(), m.clone()) for n, m in buf.views])
            b.sync_status()
            buf.check_gaps((form, K, out, mask))
        for i, ((n1, m1), (n2, m2)) in enumerate(zip(*got)):
            assert torch.equal(m1, m2) and torch.equal(n1, n2), (form, K, out, mask, i)


@pytest.mark.parametrize("form", ["pair", "quad"])
@pytest.mark.parametrize("big", [False, True])
def test_more_frames_than_the_parameter_block(form, big):
    """Aligned and other frames, empty ones among them: the run-time kernel alone, or
    strip launches of 100 frames and one launch for the rest, against the same frames
    in batches of one."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(11)
    sizes = [(64 + 8 * (i % 5) + (i % 3 == 0), 20 + i % 29 if i % 31 else 0) for i in range(230)]
    items = [(depth(W, max(H, 1), "u16" if i % 2 else "f32", gen)[:H], cameras(W, max(H, 1)))
             for i, (W, H) in enumerate(sizes)]
    if big:
        items.insert(150, (depth(2048, 2049, "u16", gen), cameras(2048, 2049)))
        items.insert(7, (depth(1920, 1081, "f32", gen), cameras(1920, 1081)))
    b = nrm.BatchedEstimator()
    one = b.multiscale(items, (1, 2, 3), form)
    two = [b.multiscale([it], (1, 2, 3), form)[0] for it in items]
    b.sync_status()
    assert_same(one, two, (form, big))
