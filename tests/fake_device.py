"""The library's host code on a stand-in device (fake_device.cpp): the C ABI
with allocations that can be counted and made to fail, without a GPU."""
import concurrent.futures as cf
import contextlib
import ctypes
import os
import shutil
import subprocess

import pytest

import paper_2111_13655_gb300 as sg
from paper_2111_13655_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
UNITS = ["sg_api.cpp", "sg_setup.cpp", "sg_rows_setup.cpp", "sg_tune.cpp", "sg_batch.cpp", "sg_solvers_api.cpp",
         "sg_server_api.cpp"]
ABSENT = ("sg_measure_peak", "sg_apply_H_noalloc")
_loaded = None


def compiler():
    """Host compiler command with CUDA's and the library's headers; skips without them."""
    cxx = shutil.which("g++") or shutil.which("c++")
    try:
        include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    except RuntimeError:
        include = ""
    if not cxx or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("needs a host C++ compiler and CUDA's headers")
    return [cxx, "-std=c++17", "-fPIC", "-isystem", include, "-I", build.CSRC, "-I", os.path.join(build.ROOT, "include")]


def load(tmp):
    """The stand-in library, built once per session into `tmp`."""
    global _loaded
    if _loaded is not None:
        return _loaded
    cxx = compiler()

    def compile_unit(path):
        obj = os.path.join(tmp, os.path.basename(path) + ".o")
        subprocess.run([*cxx, "-O1", "-c", path, "-o", obj], check=True)
        return obj

    with cf.ThreadPoolExecutor(max_workers=8) as ex:
        objs = list(ex.map(compile_unit, [os.path.join(build.CSRC, u) for u in UNITS] +
                           [os.path.join(HERE, "fake_device.cpp")]))
    so = os.path.join(tmp, "libfake.so")
    subprocess.run([cxx[0], "-shared", "-Wl,-Bsymbolic", *objs, "-o", so, "-lpthread"], check=True)
    lib = ctypes.CDLL(so)
    for name, (res, args) in sg.SIGNATURES.items():
        if name not in ABSENT:
            getattr(lib, name).restype, getattr(lib, name).argtypes = res, args
    lib.fake_fail_after.argtypes = [ctypes.c_long, ctypes.c_size_t]
    for name in ("fake_live", "fake_peak", "fake_largest"):
        getattr(lib, name).restype = ctypes.c_size_t
    for name in ("fake_matching", "fake_launches", "fake_entries"):
        getattr(lib, name).restype = ctypes.c_long
    lib.fake_launches.argtypes = [ctypes.c_char_p]
    _loaded = lib
    return lib


@contextlib.contextmanager
def use(tmp):
    """The Python binding on the stand-in library, nothing allocated and nothing failing at the start."""
    lib = load(str(tmp))
    lib.fake_reset()
    real, sg._lib = sg._lib, lib
    try:
        yield lib
    finally:
        lib.fake_fail_after(-1, 0)
        sg._lib = real
