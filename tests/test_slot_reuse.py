"""A descriptor slot whose upload is queued stays in use when a later launch of the same
call fails (host side only, on the CPU): the next call that takes the slot waits
for its event before writing the block again."""
import ctypes

import fake_gpu
from paper_2209_08241_gb300 import _lib
from test_routes import aligned, plain

SLOTS = 3


def check(call, n_launches):
    lib = fake_gpu.load()
    for fail_at in range(n_launches):
        lib.fake_reset()
        h = fake_gpu.handle(lib)
        lib.fake_fail_launch(fail_at)
        assert call(lib, h) == _lib.NRM_ERR_CUDA
        uploads = fake_gpu.log(lib).count("upload")
        for _ in range(SLOTS - 1):
            assert call(lib, h) == 0
        before = lib.fake_event_syncs()
        assert call(lib, h) == 0
        assert lib.fake_event_syncs() == before + uploads, fail_at
        lib.nrm_destroy(h)
    lib.fake_reset()


def test_forward_batches_past_the_parameter_block():
    arr = fake_gpu.frames([aligned(640, 480)] * 90 + [plain()] * 40)
    check(lambda lib, h: lib.nrm_estimate_batched(h, arr, 130, None), 2)


def test_multiscale_batches_past_the_parameter_block():
    arr = fake_gpu.frames([aligned(64, 48)] * 130)
    sc = _lib.Scales(2, (ctypes.c_int * 8)(1, 3), 0)
    check(lambda lib, h: lib.nrm_estimate_batched_multiscale(h, arr, 130, ctypes.byref(sc), None), 1)
