"""The host side of the library without a GPU: ``nrm_api.cpp`` compiled with g++
against ``fake_gpu.cpp``, whose launchers write a log. Divisions by zero and
signed overflows trap (the process dies), so calls that could contain one are
made in a child process (``in_child``)."""
import ctypes
import functools
import multiprocessing as mp
import os
import subprocess
import tempfile

from paper_2209_08241_gb300 import _lib
from paper_2209_08241_gb300 import build as nbuild

HERE = os.path.dirname(os.path.abspath(__file__))


def _compile(out):
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nbuild._nvcc()))), "include")
    flags = ["g++", "-std=c++17", "-O1", "-g", "-fPIC", "-shared", "-fvisibility=hidden", "-pthread",
             "-fsanitize=integer-divide-by-zero,signed-integer-overflow", "-fsanitize-undefined-trap-on-error",
             f"-I{cuda}", f"-I{nbuild.INCLUDE}", f"-I{nbuild.CSRC}"]
    subprocess.run(flags + [os.path.join(nbuild.CSRC, "nrm_api.cpp"), os.path.join(HERE, "fake_gpu.cpp"), "-o", out],
                   check=True)


@functools.lru_cache(None)
def _tmp():
    return tempfile.TemporaryDirectory(prefix="nrm_fake_gpu_")


@functools.lru_cache(None)
def path():
    out = os.path.join(_tmp().name, "libnrm_fake.so")
    _compile(out)
    return out


@functools.lru_cache(None)
def load(lib_path=None):
    lib = ctypes.CDLL(lib_path or path())
    for name, res, args in _lib.SIGNATURES:
        if hasattr(lib, name):
            fn = getattr(lib, name)
            fn.restype, fn.argtypes = res, args
    lib.fake_log.restype = ctypes.c_char_p
    return lib


def handle(lib, H=0, W=0, **params):
    """A handle with the default parameters but those given."""
    p = _lib.Params()
    lib.nrm_default_params(ctypes.byref(p))
    for k, v in params.items():
        setattr(p, k, v)
    h = ctypes.c_void_p()
    K = _lib.Intrinsics(500.0, 500.0, W / 2.0, H / 2.0)
    rc = lib.nrm_create(ctypes.byref(K), H, W, ctypes.byref(p), ctypes.byref(h))
    assert rc == 0, lib.nrm_last_error()
    return h


BASE = 1 << 20  # of every buffer: nothing reads or writes them


def frames(specs):
    """specs: (W, H, in_dtype, depth pitch, out pitch, offset of normals in bytes)"""
    arr = (_lib.Frame * max(len(specs), 1))()
    for f, (W, H, dtype, dp, op, off) in zip(arr, specs):
        f.depth, f.normals, f.valid = BASE, BASE + off, BASE
        f.H, f.W, f.depth_pitch, f.out_pitch, f.in_dtype = H, W, dp, op, dtype
        f.K = _lib.Intrinsics(500.0, 500.0, W / 2.0, H / 2.0)
    return arr


def grad_frames(specs):
    """specs: (W, H)"""
    arr = (_lib.GradFrame * max(len(specs), 1))()
    for f, (W, H) in zip(arr, specs):
        f.depth = f.grad_normals = f.valid = f.grad_depth = BASE
        f.H, f.W, f.depth_pitch, f.out_pitch = H, W, W, W
        f.K = _lib.Intrinsics(500.0, 500.0, W / 2.0, H / 2.0)
    return arr


def log(lib):
    """The launches (and uploads) since the last reset, one line each."""
    return lib.fake_log().decode().splitlines()


def in_child(target, *args):
    """Exit code of target(*args) in a process of its own."""
    p = mp.get_context("spawn").Process(target=target, args=args)
    p.start()
    p.join(120)
    return p.exitcode
