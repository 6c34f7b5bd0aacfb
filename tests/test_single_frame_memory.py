"""nrm_estimate allocates no host memory, whichever kernel takes the frame (host side
only, on the CPU, in a process whose allocations fail during the call: an
allocation's exception would end it at the C boundary)."""
import pytest

import fake_gpu


def _estimate(lib_path, H, W, out, offset):
    lib = fake_gpu.load(lib_path)
    h = fake_gpu.handle(lib, H, W, out_dtype=out)
    B = fake_gpu.BASE
    lib.fake_no_memory(1)
    rc = lib.nrm_estimate(h, B, B + offset, B, None)
    lib.fake_no_memory(0)
    assert rc == 0 and len(fake_gpu.log(lib)) == 1


@pytest.mark.parametrize("H,W,out,offset", [(480, 640, 0, 0), (3072, 4096, 0, 0), (3071, 4095, 2, 4)])
def test_no_host_allocation(H, W, out, offset):
    assert fake_gpu.in_child(_estimate, fake_gpu.path(), H, W, out, offset) == 0
