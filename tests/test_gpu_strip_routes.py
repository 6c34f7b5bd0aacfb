"""The forward kernels of batched calls against one another, on batches that reach each
of them (tests/test_routes.py checks on the CPU which ones these reach): the strip
kernel for aligned frames, the one for any alignment, and two launches, each bit
for bit equal to the tiled kernels. Outputs lie in buffers with gaps between the
rows and around them, which must keep their contents."""
import pytest
import torch

import paper_2209_08241_gb300 as nrm
from test_gpu_strip import DEV, bits, depth

pytestmark = pytest.mark.gpu
# (W, H): batches of these in float32, and in uint16 where the rows are whole 16-byte units.
ALIGNED = [(4, 1), (8, 5), (124, 23), (128, 24), (136, 25), (256, 31), (264, 33), (640, 49), (1032, 97)]
# (W, H, gap behind a row, first pixel of the outputs): the last frame makes the batch large enough.
ANY = [(1, 1, 0, 1), (3, 2, 1, 0), (5, 24, 2, 3), (127, 25, 0, 0), (129, 23, 1, 2), (131, 49, 5, 0), (255, 33, 0, 1),
       (257, 5, 3, 3), (128, 24, 3, 1), (389, 47, 1, 0), (1601, 1201, 2, 1)]
OUT = {"f32": (torch.float32, 4), "f16": (torch.float16, 4), "oct16": (torch.int16, 2)}
SENT = 77


class Buffers:
    """Normals and mask of each frame inside larger buffers of a fixed byte."""

    def __init__(self, items, out, gaps):
        dt, C = OUT[out]
        self.raw, self.views = [], []
        for (d, _), (pad, start) in zip(items, gaps):
            H, W = d.shape
            P = W + pad
            n = torch.full(((H * P + start + 8) * C * dt.itemsize,), SENT, dtype=torch.uint8, device=DEV)
            v = torch.full((H * P + start + 8,), SENT, dtype=torch.uint8, device=DEV)
            nv = n.view(dt)[start * C:(start + H * P) * C].view(H, P, C)[:, :W]
            self.raw.append((n, v))
            self.views.append((nv, v[start:start + H * P].view(H, P)[:, :W]))

    def check_gaps(self, what):
        for i, ((n, v), (nv, vv)) in enumerate(zip(self.raw, self.views)):
            nv.view(torch.uint8).fill_(SENT)
            vv.fill_(SENT)
            assert bool((n == SENT).all()) and bool((v == SENT).all()), (what, i)


def compare(b, items, out, gaps, what):
    got = []
    for config in ((128, 16, 256, 3, 0), (128, 8, 128, 2, 0)):
        b.set_config(*config)
        buf = Buffers(items, out, gaps)
        b(items, buf.views)
        got.append([(bits(n).clone(), m.clone()) for n, m in buf.views])
        b.sync_status()
        buf.check_gaps((what, config))
    for i, ((n1, m1), (n2, m2)) in enumerate(zip(*got)):
        assert torch.equal(m1, m2) and torch.equal(n1, n2), (what, i)


def cameras(W, H):
    return (0.8 * W, 0.9 * W, 0.4 * W, 0.6 * H)


@pytest.mark.parametrize("out", OUT)
@pytest.mark.parametrize("alpha", [1, 2, 3, 4])
@pytest.mark.parametrize("mask", ["secant", "raw"])
def test_aligned_frames(out, alpha, mask):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(alpha)
    items = [(depth(W, H, t, gen), cameras(W, H)) for W, H in ALIGNED for t in ("f32", "u16")
             if W * (2 if t == "u16" else 4) % 16 == 0]
    for sign in (False, True):
        b = nrm.BatchedEstimator(nrm.NormalParams(alpha=alpha, out_dtype=out, mask_mode=mask, orient_to_camera=sign,
                                                  tau=12.0 if mask == "secant" else 1e-3))
        # Rows of outputs 8 pixels longer than the frame, starting 8 pixels into the buffer.
        compare(b, items, out, [(8 * (i % 2), 8) for i in range(len(items))], (out, alpha, mask, sign))
        u16 = [it for it in items if it[0].dtype == torch.uint16]
        compare(b, u16, out, [(0, 0)] * len(u16), (out, alpha, mask, sign, "u16 only"))


@pytest.mark.parametrize("out", OUT)
@pytest.mark.parametrize("alpha", [1, 2, 3, 4])
@pytest.mark.parametrize("times", [1, 5])
def test_frames_of_any_alignment(out, alpha, times):
    """times 5: 110 frames, past the parameter block."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(alpha)
    items, gaps = [], []
    for W, H, pad, start in ANY:
        for t in ("f32", "u16"):
            d = depth(W + pad, H, t, gen)[:, :W]
            items.append((d, cameras(W, H)))
            gaps.append((pad, start))
    for mask, tau in (("secant", 12.0), ("raw", 1e-3)):
        b = nrm.BatchedEstimator(nrm.NormalParams(alpha=alpha, out_dtype=out, mask_mode=mask, tau=tau))
        compare(b, items * times, out, gaps * times, (out, alpha, mask))


@pytest.mark.parametrize("out", OUT)
def test_two_launches_and_one(out):
    """Aligned and other frames: enough of both for two launches, then a few small
    ones, then ragged frames (which TMA loads) of widths not in fours."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(5)
    big = [(depth(1920, 1080, "u16", gen), cameras(1920, 1080)) for _ in range(8)]
    odd = [(depth(1921, 1081, "u16", gen), cameras(1921, 1081)) for _ in range(8)]
    ragged = [(depth(1920, 1078, "u16", gen)[:, :1917], cameras(1917, 1078)) for _ in range(4)]
    for alpha in (1, 2, 4):
        b = nrm.BatchedEstimator(nrm.NormalParams(alpha=alpha, out_dtype=out))
        compare(b, big * 4 + odd, out, [(0, 0)] * 40, (out, alpha, "two launches"))
        compare(b, ragged, out, [(1, 0), (0, 1), (3, 0), (2, 3)], (out, alpha, "ragged"))
        small = [(d[:200, :256].contiguous(), cameras(256, 200)) for d, _ in big[:3]] + [
            (d[:101, :133].contiguous(), cameras(133, 101)) for d, _ in odd[:3]]
        compare(b, small, out, [(0, 0)] * 6, (out, alpha, "small"))
