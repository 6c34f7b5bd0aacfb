"""The range-checking build (see test_gpu_checked_build.py) over the tests of the strip,
multi-scale strip, adjoint, evaluation, loss-scale and plane-fit kernels."""
import os
import subprocess
import sys

import pytest

from paper_2209_08241_gb300 import build as nbuild

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SELECTION = [
    "tests/test_gpu_strip_routes.py",
    "tests/test_gpu_strip.py::test_large_single_frames_same_bits_as_the_plain_kernel",
    "tests/test_gpu_multiscale_routes.py",
    "tests/test_gpu_adjoint_tiles.py",
    "tests/test_gpu_adjoint_forms.py",
    "tests/test_gpu_adjoint_distances.py",
    "tests/test_gpu_mse_pieces.py",
    "tests/test_gpu_mse_images.py",
    "tests/test_gpu_loss_scale.py",
    "tests/test_gpu_loss_scale_wide.py",
    "tests/test_gpu_plane_fit_forms.py",
]


def test_checked_build_passes_the_tests_of_these_kernels():
    nbuild.build(debug=True)
    env = dict(os.environ, NRM_LIB_VARIANT="debug")
    cmd = [sys.executable, "-m", "pytest", "-q", "-x", "-m", "gpu", "-p", "no:cacheprovider", "-s", *SELECTION]
    out = subprocess.run(cmd, cwd=ROOT, env=env, capture_output=True, text=True, timeout=3000)
    text = out.stdout + out.stderr
    bad = [ln for ln in text.splitlines() if "NRM_BOUNDS" in ln]
    assert not bad, "\n".join(bad)[:4000]
    assert out.returncode == 0, text[-4000:]
    assert " passed" in text and " failed" not in text
