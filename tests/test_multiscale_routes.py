"""Which kernel a batched multi-scale call's frames go to (host side only, on the CPU):
the strip kernel for consecutive distances, aligned frames and enough tiles of
them, else the run-time-distance kernel, in one launch where the strip kernel
does not pay for a second one."""
import ctypes

import pytest

import fake_gpu
from paper_2209_08241_gb300 import _lib
from test_routes import F32, OUTS, aligned, plain, ragged


def launches(specs, alphas, form="pair", out="f32", capture=0, **params):
    lib = fake_gpu.load()
    lib.fake_reset()
    h = fake_gpu.handle(lib, out_dtype=OUTS[out], **params)
    lib.fake_capture(capture)
    sc = _lib.Scales(len(alphas), (ctypes.c_int * 8)(*alphas), {"pair": 0, "quad": 1}[form])
    rc = lib.nrm_estimate_batched_multiscale(h, fake_gpu.frames(specs), len(specs), ctypes.byref(sc), None)
    assert rc == 0, lib.nrm_last_error()
    lines = fake_gpu.log(lib)
    lib.fake_reset()
    lib.nrm_destroy(h)
    return [(w[0], int(w[1].split("=")[1])) for w in (ln.split() for ln in lines) if w[0] != "upload"]


@pytest.mark.parametrize("form", ["pair", "quad"])
@pytest.mark.parametrize("K", [2, 4, 6])
def test_aligned_batches(form, K):
    alphas = range(1, K + 1)
    for n, W, H in ((1, 160, 120), (1, 640, 480), (2, 640, 480), (16, 64, 48)):
        assert launches([aligned(W, H)] * n, alphas, form) == [("ms_tiled", n)]
    for n, W, H in ((16, 640, 480), (16, 1920, 1080), (1, 4096, 3072)):
        assert launches([aligned(W, H, F32)] * n, alphas, form) == [("ms_strip", n)]
    few = "ms_tiled" if form == "quad" and K == 6 else "ms_strip"
    assert launches([aligned(1280, 720)], alphas, form, "f16") == [(few, 1)]
    assert launches([aligned(640, 480)] * 4, alphas, form, "oct16") == [(few, 4)]


@pytest.mark.parametrize("capture", [0, 1])
@pytest.mark.parametrize("other", [plain, ragged])
def test_mixed_batches(capture, other):
    for batch in ([aligned(), other()], [aligned()] * 7 + [other()], [aligned()] + [other()] * 7,
                  [aligned(1920, 1080), other()]):
        assert launches(batch, range(1, 5), "pair", capture=capture) == [("ms_tiled", len(batch))]
    batch = [aligned(1920, 1080)] * 4 + [other(1921, 1081)] * 4
    assert launches(batch, (1, 2), "pair", capture=capture) == [("ms_tiled", 8)]
    assert launches(batch, (1, 2), "quad", capture=capture) == [("ms_strip", 4), ("ms_tiled", 4)]
    batch = [aligned(1920, 1080)] * 7 + [other()]
    assert launches(batch, range(1, 5), "quad", capture=capture) == [("ms_strip", 7), ("ms_tiled", 1)]


def test_batches_past_the_parameter_block():
    """The run-time kernel takes any number of frames in one launch, the strip kernel
    100 a launch."""
    assert launches([aligned(64, 48)] * 256, (1, 3)) == [("ms_tiled", 256)]
    assert launches([aligned(64, 48)] * 256, range(1, 5)) == [("ms_tiled", 256)]
    assert launches([plain(65, 49)] * 101, range(1, 5)) == [("ms_tiled", 101)]
    assert launches([aligned()] * 130, range(1, 5)) == [("ms_strip", 100), ("ms_strip", 30)]
    assert launches(([aligned()] * 2 + [plain()]) * 60, range(1, 5)) == [("ms_strip", 100), ("ms_strip", 20),
                                                                        ("ms_tiled", 60)]


def test_other_distances_and_frames():
    big = [aligned(1920, 1080)] * 4
    for alphas in ((1, 3), (2, 1), (1,), (2, 3, 4), range(1, 8), range(1, 9)):
        assert launches(big, alphas) == [("ms_tiled", 4)]
    assert launches([plain(1921, 1081)] * 4, range(1, 5)) == [("ms_tiled", 4)]
    assert launches(big, range(1, 5), depth_scale=1e-9) == [("ms_tiled", 4)]


@pytest.mark.parametrize("form", ["pair", "quad"])
def test_the_bit_comparisons_reach_the_strip_kernel(form):
    """The batches of test_gpu_multiscale_routes.py."""
    import test_gpu_multiscale_routes as gpu
    eb = {"f32": 4, "u16": 2}
    for K in range(2, 7):
        batch = [aligned(W, H, F32 if t == "f32" else 1) for W, H in gpu.SIZES for t in eb if W * eb[t] % 16 == 0]
        assert launches(batch, range(1, K + 1), form) == [("ms_strip", len(batch))]
        times = -(-101 // len(batch))
        got = launches(batch * times, range(1, K + 1), form)
        assert {k for k, _ in got} == {"ms_strip"} and sum(n for _, n in got) == len(batch) * times
        small = [aligned(W, H) for W, H in gpu.SMALL]
        assert launches(small, range(1, K + 1), form) == [("ms_tiled", len(small))]
