"""What the autotune cache's keys keep apart (host side only, on the CPU): entries timed
on older kernels, and geometries tuned for point clouds, which say nothing about
the kernels that calls without point clouds take."""
import ctypes
import json

import pytest

import fake_gpu
from paper_2209_08241_gb300 import _lib
from test_routes import F32, aligned

TILED = {"tile_x": 128, "tile_y": 16, "threads": 256, "stages": 2, "ctas_per_sm": 2}  # the second candidate


@pytest.fixture
def lib(tmp_path):
    lib = fake_gpu.load()
    lib.fake_reset()
    path = str(tmp_path / "tune.json").encode()
    assert lib.nrm_set_autotune_cache(path) == 0
    lib.cache_file = path
    yield lib
    lib.nrm_set_autotune_cache(None)
    lib.fake_reset()


def batch(points=False, n=3):
    arr = fake_gpu.frames([aligned(640, 480, F32)] * n)
    for f in arr:
        f.points = fake_gpu.BASE if points else None
    return arr


def tune(lib, h, points=False, fastest=-1):
    """Tunes the handle; the number of candidates that were timed."""
    lib.fake_reset()
    lib.fake_fastest(fastest)
    assert lib.nrm_autotune(h, batch(points), 3, None, None) == 0, lib.nrm_last_error()
    return lib.fake_timings()


def config(lib, h):
    c = _lib.TileConfig()
    assert lib.nrm_get_config(h, ctypes.byref(c)) == 0
    return {name: getattr(c, name) for name, _ in c._fields_}


def kernel(lib, h):
    """The kernel of a batch without point clouds."""
    lib.fake_reset()
    assert lib.nrm_estimate_batched(h, batch(), 3, None) == 0
    return fake_gpu.log(lib)[0].split()[0]


def test_the_strip_kernels_stay_when_they_are_the_fastest(lib):
    h = fake_gpu.handle(lib)
    assert tune(lib, h) > 1 and kernel(lib, h) == "strip"
    assert tune(lib, h) == 0 and kernel(lib, h) == "strip"  # from the cache
    assert kernel(lib, fake_gpu.handle(lib)) == "strip"


def test_a_faster_tiled_geometry_is_kept(lib):
    h = fake_gpu.handle(lib)
    assert tune(lib, h, fastest=1) > 1
    assert config(lib, h) == TILED and kernel(lib, h) == "tiled"
    other = fake_gpu.handle(lib)  # picks the handle's entry up
    assert config(lib, other) == TILED and kernel(lib, other) == "tiled"
    assert tune(lib, other) == 0 and kernel(lib, other) == "tiled"


def test_entries_of_older_kernels_are_not_used(lib):
    h = fake_gpu.handle(lib)
    tune(lib, h, fastest=1)
    entries = json.load(open(lib.cache_file))
    old = {k.replace("|k2|", "|"): v for k, v in entries.items()}
    assert len(entries) == 2 and not set(old) & set(entries)
    json.dump(old, open(lib.cache_file, "w"))
    h = fake_gpu.handle(lib)
    assert kernel(lib, h) == "strip" and config(lib, h)["ctas_per_sm"] == 0
    assert tune(lib, h) > 1 and kernel(lib, h) == "strip"


def test_tuning_for_point_clouds_leaves_other_calls_alone(lib):
    h = fake_gpu.handle(lib)
    assert tune(lib, h, points=True, fastest=1) > 1
    assert config(lib, h) == TILED and kernel(lib, h) == "strip"
    assert tune(lib, h, points=True) == 0 and kernel(lib, h) == "strip"
    other = fake_gpu.handle(lib)
    assert config(lib, other) == TILED and kernel(lib, other) == "strip"
    assert tune(lib, other) > 1 and kernel(lib, other) == "strip"  # no entry without point clouds yet
    # An explicit geometry decides for both.
    assert lib.nrm_set_config(h, ctypes.byref(_lib.TileConfig(**TILED))) == 0
    assert kernel(lib, h) == "tiled"
    assert tune(lib, h, points=True) == 0 and kernel(lib, h) == "tiled"
    assert lib.nrm_set_config(h, ctypes.byref(_lib.TileConfig(128, 16, 256, 3, 0))) == 0
    assert kernel(lib, h) == "strip"


def test_a_failed_sweep_restores_the_handle(lib):
    h = fake_gpu.handle(lib)
    lib.fake_reset()
    lib.fake_fail_launch(9)
    assert lib.nrm_autotune(h, batch(), 3, None, None) == _lib.NRM_ERR_CUDA
    assert config(lib, h)["ctas_per_sm"] == 0 and kernel(lib, h) == "strip"
