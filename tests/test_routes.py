"""Which kernels a call's frames go to and in how many launches (host side only, on the
CPU): batches of one kind of frame and of several, with the parameter block and the
descriptor ring, under capture, and single frames. "Aligned" frames are those
that the strip kernel with vector stores takes, "ragged" ones others that TMA
can load, "plain" ones have rows that it cannot."""
import ctypes

import pytest

import fake_gpu
from paper_2209_08241_gb300 import _lib

F32, U16 = _lib.NRM_IN_F32_M, _lib.NRM_IN_U16_MM
OUTS = {"f32": 0, "f16": 1, "oct16": 2}


def aligned(W=640, H=480, dtype=U16):
    return (W, H, dtype, W, W, 0)


def ragged(W=638, H=478, dtype=U16, out_pitch=None, offset=0):
    return (W, H, dtype, (W + 7) // 8 * 8, out_pitch or W, offset)


def plain(W=641, H=481, dtype=U16):
    return (W, H, dtype, W, W, 0)


def launches(specs, out="f32", capture=0, config=None, **params):
    lib = fake_gpu.load()
    lib.fake_reset()
    h = fake_gpu.handle(lib, out_dtype=OUTS[out], **params)
    if config:
        assert lib.nrm_set_config(h, ctypes.byref(_lib.TileConfig(*config))) == 0
    lib.fake_capture(capture)
    rc = lib.nrm_estimate_batched(h, fake_gpu.frames(specs), len(specs), None)
    assert rc == 0, lib.nrm_last_error()
    lines = fake_gpu.log(lib)
    lib.fake_reset()
    lib.nrm_destroy(h)
    return [(w[0], int(w[1].split("=")[1])) for w in (ln.split() for ln in lines) if w[0] != "upload"]


@pytest.mark.parametrize("out", OUTS)
@pytest.mark.parametrize("n", [1, 3, 100, 130])
@pytest.mark.parametrize("alpha", [1, 2, 3, 4])
def test_aligned_batches_take_the_aligned_strip_kernel(out, n, alpha):
    for W, H in ((4, 1), (64, 48), (640, 480), (1920, 1080)):
        assert launches([aligned(W, H, F32)] * n, out, alpha=alpha) == [("strip", n)]
    assert launches([aligned()] * n, out, alpha=alpha) == [("strip", n)]


@pytest.mark.parametrize("out", OUTS)
def test_other_geometries_and_distances_take_the_tiled_kernel(out):
    batch = [aligned(), plain(), ragged()]
    assert launches(batch, out, alpha=5) == [("tiled", 3)]
    assert launches(batch, out, config=(128, 8, 128, 2, 0)) == [("tiled", 3)]
    assert launches(batch, out, config=(128, 16, 256, 3, 2)) == [("tiled", 3)]


@pytest.mark.parametrize("out", OUTS)
@pytest.mark.parametrize("capture", [0, 1])
def test_small_mixed_batches_take_one_launch(out, capture):
    for batch in ([aligned(), plain()], [aligned(320, 240)] * 4 + [plain(321, 241)] * 4, [aligned()] + [plain()] * 7,
                  [aligned(320, 240)] * 7 + [plain(321, 241)], [aligned(), ragged()], [aligned()] + [ragged()] * 15):
        got = launches(batch, out, capture)
        assert len(got) == 1 and got[0][1] == len(batch), (batch, got)


@pytest.mark.parametrize("out", OUTS)
@pytest.mark.parametrize("capture", [0, 1])
@pytest.mark.parametrize("n,m", [(31, 1), (16, 16)])
def test_large_mixed_batches_take_two_launches(out, capture, n, m):
    batch = [aligned(1920, 1080)] * n + [plain(1921, 1081)] * m
    assert launches(batch, out, capture) == [("strip", n), ("strip_any", m)]


@pytest.mark.parametrize("alpha", [1, 2])
def test_ragged_frames_take_the_cheaper_kernel(alpha):
    """Half4 tiles have vector loops at alpha 1 and 2; so have octahedral ones with rows
    of codes on 16 bytes. Float4 frames of some size are cheaper without."""
    for n in (1, 16, 64):
        assert launches([ragged(1918, 1078)] * n, "f16", alpha=alpha) == [("tiled", n)]
        assert launches([ragged(1918, 1078, F32, 1920)] * n, "f16", alpha=alpha) == [("tiled", n)]
    assert launches([ragged(1918, 1078, U16, 1920)] * 64, "oct16", alpha=2) == [("tiled", 64)]
    assert launches([ragged(1918, 1078)] * 64, "oct16", alpha=alpha) == [("strip_any", 64)]
    assert launches([ragged(1918, 1078)] * 64, "f32", alpha=alpha) == [("strip_any", 64)]
    for out in OUTS:
        assert launches([ragged(318, 238)], out, alpha=alpha) == [("tiled", 1)]


@pytest.mark.parametrize("out", OUTS)
def test_plain_frames(out):
    assert launches([plain()] * 16, out) == [("strip_any", 16)]
    assert launches([plain(1921, 1081)] * 130, out) == [("strip_any", 130)]
    # (A depth scale at which q may fall below FLT_MIN keeps uint16 frames on the tiled kernel.)
    assert launches([plain()] * 16 + [aligned()], out, depth_scale=1e-9) == [("tiled", 17)]


def test_ring_batches_of_both_kinds():
    assert launches([aligned(640, 480)] * 90 + [plain()] * 40) == [("strip", 90), ("strip_any", 40)]
    assert launches([aligned(64, 48)] * 90 + [plain(65, 49)] * 40) == [("strip_any", 130)]


@pytest.mark.parametrize("out", OUTS)
@pytest.mark.parametrize("W,H,offset,want", [
    (640, 480, 0, "plain"), (2000, 1504, 0, "strip"), (4096, 3072, 0, "strip"), (4095, 3071, 0, "strip_any"),
    (2001, 1503, 0, "strip_any or plain"), (2048, 1536, 16, "unaligned outputs")])
def test_single_frames(out, W, H, offset, want):
    lib = fake_gpu.load()
    lib.fake_reset()
    h = fake_gpu.handle(lib, H, W, out_dtype=OUTS[out], in_dtype=U16)
    offset = {"f32": 16, "f16": 8, "oct16": 4}[out] if offset else 0
    B = fake_gpu.BASE
    assert lib.nrm_estimate(h, B, B + offset, B, None) == 0
    got = [ln.split()[0] for ln in fake_gpu.log(lib)]
    lib.nrm_destroy(h)
    if want == "strip_any or plain":
        want = "plain" if out == "f16" else "strip_any"
    if want == "unaligned outputs":
        want = "strip_any" if out == "f32" else "plain"
    assert got == [want]


@pytest.mark.parametrize("out", OUTS)
@pytest.mark.parametrize("alpha", [1, 2, 3, 4])
def test_the_bit_comparisons_reach_the_kernels_they_are_for(out, alpha):
    """The batches of test_gpu_strip_routes.py."""
    import test_gpu_strip_routes as gpu
    eb = {F32: 4, U16: 2}

    def spec(W, H, dtype, pad, start):
        return (W, H, dtype, W + pad, W + pad, start * {"f32": 16, "f16": 8, "oct16": 4}[out])

    batch = [spec(W, H, t, 0, 0) for W, H in gpu.ALIGNED for t in (F32, U16) if W * eb[t] % 16 == 0]
    assert launches(batch, out, alpha=alpha) == [("strip", len(batch))]
    batch = [spec(W, H, t, pad, start) for W, H, pad, start in gpu.ANY for t in (F32, U16)]
    assert launches(batch, out, alpha=alpha) == [("strip_any", len(batch))]
    batch = batch * 5
    assert launches(batch, out, alpha=alpha) == [("strip_any", len(batch))]
    batch = [aligned(1920, 1080)] * 32 + [plain(1921, 1081)] * 8
    assert launches(batch, out, alpha=alpha) == [("strip", 32), ("strip_any", 8)]
