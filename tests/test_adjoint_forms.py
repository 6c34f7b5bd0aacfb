"""Every distance that the adjoint accepts reaches its launch, in the single and the
batched entry points (host side only, on the CPU): the form with weights in
registers exists for distances 2 to 4 alone, and at 16 its tile would be
empty."""
import sys

import pytest

import fake_gpu
from paper_2209_08241_gb300 import _lib


def _adjoint(lib_path, W, H, n):
    lib = fake_gpu.load(lib_path)
    arr = fake_gpu.grad_frames([(W, H)] * n)
    B = fake_gpu.BASE
    for alpha in range(1, _lib.NRM_MAX_ALPHA + 1):
        print("alpha", alpha, file=sys.stderr, flush=True)
        lib.fake_reset()
        h = fake_gpu.handle(lib, H, W, alpha=alpha)
        assert lib.nrm_backward(h, B, B, B, B, None) == 0
        assert lib.nrm_backward_batched(h, arr, n, None) == 0
        launches = [ln.split() for ln in fake_gpu.log(lib) if ln != "upload"]
        assert [ln[0] for ln in launches] == ["bwd", "bwd_batch" if n <= 60 else "bwd_ring"]
        if alpha not in (2, 3, 4):
            assert all("walk=0" in ln for ln in launches)
        lib.nrm_destroy(h)


@pytest.mark.parametrize("W,H,n", [(640, 480, 3), (97, 31, 70), (1, 1, 1)])
def test_every_distance_reaches_its_launch(W, H, n):
    assert fake_gpu.in_child(_adjoint, fake_gpu.path(), W, H, n) == 0
