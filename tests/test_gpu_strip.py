"""The strip kernels (batched forward with the default geometry) against the
tiled kernels (any other geometry): the same bits, over widths and heights
around the tile edges, every pixel distance they are compiled for, both input
types, all outputs, both mask modes, depth values of every kind, frames of any
alignment, batches past the parameter block and batches of both kinds."""
import pytest
import torch

import paper_2209_08241_gb300 as nrm

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SIZES = [(4, 1), (8, 5), (124, 23), (128, 24), (132, 25), (256, 31), (260, 33), (640, 49), (1028, 97)]


def depth(W, H, dtype, gen):
    z = 2.0 + 0.02 * torch.randn((H, W), generator=gen, device=DEV) + torch.rand((H, 1), generator=gen, device=DEV)
    z[torch.rand((H, W), generator=gen, device=DEV) < 0.03] *= 2.0
    bad = torch.rand((H, W), generator=gen, device=DEV) < 0.03
    if dtype == "u16":
        z = torch.where(bad, 0.0, (z * 1000.0).round())
        z[torch.rand((H, W), generator=gen, device=DEV) < 0.01] = 65535.0
        return z.to(torch.int32).to(torch.uint16)
    odd = torch.tensor([0.0, -0.0, -1.5, float("inf"), -float("inf"), float("nan"), 1e-40, 1e-30, 3e38], device=DEV)
    pick = torch.randint(0, len(odd), (H, W), generator=gen, device=DEV)
    return torch.where(bad, odd[pick], z)


def both(b, items, outputs=lambda: None):
    """The batch through the strip kernels and through the tiled ones."""
    b.set_config(128, 16, 256, 3, 0)
    one = b(items, outputs=outputs())
    b.set_config(128, 8, 128, 2, 0)
    two = b(items, outputs=outputs())
    b.sync_status()
    return one, two


def bits(t):
    t = t.contiguous()
    return t.view(torch.int32) if t.dtype == torch.float32 else t.view(torch.int16)


def assert_same(one, two, what):
    for i, ((n1, m1), (n2, m2)) in enumerate(zip(one, two)):
        assert torch.equal(m1, m2), (what, i)
        assert torch.equal(bits(n1), bits(n2)), (what, i)


@pytest.mark.parametrize("out", ["f32", "f16", "oct16"])
@pytest.mark.parametrize("alpha", [1, 2, 3, 4])
@pytest.mark.parametrize("mask", ["secant", "raw"])
def test_same_bits_as_the_tiled_kernels(out, alpha, mask):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(alpha)
    for sign in (False, True):
        b = nrm.BatchedEstimator(nrm.NormalParams(alpha=alpha, out_dtype=out, mask_mode=mask, orient_to_camera=sign,
                                                  tau=12.0 if mask == "secant" else 1e-3))
        items = [(depth(W, H, dt, gen), (0.8 * W, 0.9 * W, 0.4 * W, 0.6 * H)) for W, H in SIZES for dt in ("f32", "u16")]
        assert_same(*both(b, items), (out, alpha, mask, sign))
        assert_same(*both(b, items[1::2]), (out, alpha, mask, sign, "u16 only"))


@pytest.mark.parametrize("out", ["f32", "f16", "oct16"])
@pytest.mark.parametrize("alpha", [1, 2, 3, 4])
def test_any_alignment_same_bits_as_the_tiled_kernels(out, alpha):
    """Frames that TMA cannot load (odd widths and pitches, depth starting on any
    element), outputs of every alignment."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(alpha)
    C, dt = (2, torch.int16) if out == "oct16" else (4, torch.float16 if out == "f16" else torch.float32)
    sizes = [(1, 1), (3, 2), (5, 24), (127, 25), (129, 23), (131, 49), (255, 33), (257, 5), (389, 47)]
    for mask, tau in (("secant", 12.0), ("raw", 1e-3)):
        b = nrm.BatchedEstimator(nrm.NormalParams(alpha=alpha, out_dtype=out, mask_mode=mask, tau=tau))
        items, starts = [], []
        for i, (W, H) in enumerate(sizes):
            for dtype in ("f32", "u16"):
                d = depth(W + 2, H, dtype, gen)[:, i % 3:i % 3 + W]
                items.append((d, (0.8 * W, 0.9 * W, 0.4 * W, 0.6 * H)))
                starts.append(i % 4)

        def outputs():
            made = []
            for (d, _), s in zip(items, starts):
                H, W = d.shape
                nb = torch.zeros((H * (W + s) + s, C), dtype=dt, device=DEV)[s:].view(H, W + s, C)
                vb = torch.zeros(H * (W + s) + s, dtype=torch.uint8, device=DEV)[s:].view(H, W + s)
                made.append((nb[:, :W], vb[:, :W]))
            return made

        assert_same(*both(b, items, outputs), (out, alpha, mask))


@pytest.mark.parametrize("out", ["f32", "oct16"])
def test_large_and_partly_eligible_batches(out):
    """More frames than the parameter block takes (one upload, two launches), a
    third of them of widths or pitches that the strip kernels do not take,
    empty frames among them; then more tiles than one wave."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(9)
    C, dt = (2, torch.int16) if out == "oct16" else (4, torch.float32)
    sizes = [(64 + 4 * (i % 7) + (i % 3 == 0), 20 + i % 29 if i % 31 else 0) for i in range(130)]
    items = [(depth(W, max(H, 1), "u16" if i % 2 else "f32", gen)[:H], (60.0, 70.0, 30.0, 20.0))
             for i, (W, H) in enumerate(sizes)]

    def outputs():
        pads = [1 if i % 5 == 0 else 8 for i in range(len(sizes))]
        return [(torch.zeros((H, W + p, C), dtype=dt, device=DEV)[:, :W],
                 torch.zeros((H, W + p), dtype=torch.uint8, device=DEV)[:, :W]) for (W, H), p in zip(sizes, pads)]

    b = nrm.BatchedEstimator(nrm.NormalParams(out_dtype=out))
    assert_same(*both(b, items, outputs), (out, "ring"))
    assert_same(*both(b, items[:40], outputs), (out, "parameter block"))
    big = [(depth(1920, 1083, "u16", gen), (1500.0, 1500.0, 960.0, 540.0)) for _ in range(9)]
    assert_same(*both(b, big), (out, "several waves"))


def test_uint16_frames_whose_statistic_could_underflow_take_the_tiled_kernels():
    """With a depth scale so small that q of a valid pixel falls below FLT_MIN the
    pixel is masked (the documented domain); the strip kernels leave that
    test out, so such frames must not go there."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(3)
    b = nrm.BatchedEstimator(nrm.NormalParams(depth_scale=1e-9))
    items = [(torch.randint(1, 40, (64, 256), generator=gen, device=DEV).to(torch.uint16), (500.0, 500.0, 128.0, 32.0))]
    one, two = both(b, items)
    assert_same(one, two, "underflow")


@pytest.mark.parametrize("form", ["pair", "quad"])
@pytest.mark.parametrize("K", [2, 3, 4, 5, 6])
def test_multiscale_same_bits_as_the_run_time_distance_kernel(form, K):
    """Distances 1..K: frames with aligned rows take the strip kernels, the same
    frames with an odd output pitch the other kernel. More frames than one
    launch takes, sizes around the tile edges, depth values of every kind."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(K)
    sizes = SIZES + [(64, 63), (128, 64), (136, 65), (384, 7)]
    items = [(depth(W, H, dt, gen), (0.8 * W, 0.9 * W, 0.4 * W, 0.6 * H)) for W, H in sizes for dt in ("f32", "u16")]
    items = items * 5 if K == 4 else items
    for out, C, dt in (("f32", 4, torch.float32), ("f16", 4, torch.float16), ("oct16", 2, torch.int16)):
        for mask, tau in (("secant", 12.0), ("raw", 1e-3)):
            b = nrm.BatchedEstimator(nrm.NormalParams(out_dtype=out, mask_mode=mask, tau=tau))
            wide = [(torch.zeros((*d.shape[:1], d.shape[1] + 1, C), dtype=dt, device=DEV)[:, :d.shape[1]],
                     torch.zeros((d.shape[0], d.shape[1] + 1), dtype=torch.uint8, device=DEV)[:, :d.shape[1]])
                    for d, _ in items]
            one = b.multiscale(items, range(1, K + 1), form)
            two = b.multiscale(items, range(1, K + 1), form, outputs=wide)
            b.sync_status()
            assert_same(one, two, (form, K, out, mask))


@pytest.mark.parametrize("W,H", [(2400, 1251), (1999, 1503), (4096, 735)])
@pytest.mark.parametrize("dtype,out", [("f32", "f32"), ("u16", "f16"), ("u16", "oct16")])
def test_large_single_frames_same_bits_as_the_plain_kernel(W, H, dtype, out):
    """Single-frame calls of three million pixels and more take the strip kernels."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(W)
    d = depth(W, H, dtype, gen)
    est = nrm.NormalEstimator((0.8 * W, 0.9 * W, 0.4 * W, 0.6 * H), H, W, nrm.NormalParams(out_dtype=out), dtype)
    one = est.estimate(d)
    est.set_config(128, 8, 128, 2, 0)
    two = est.estimate(d)
    est.sync_status()
    assert_same([one], [two], (W, H, dtype, out))
