"""The library's C API over a stand-in for the CUDA runtime and the kernels'
launchers (fake_device.cpp), for CPU tests of what sq_api.cpp decides: what goes
into a launch, how calls on several streams are ordered, what a failing call
leaves behind."""
import ctypes
import os
import shutil
import subprocess

from paper_2602_22603_gb300 import build, _SIGS

HERE = os.path.dirname(os.path.abspath(__file__))
APPEND, APPEND_BATCH, DECODE, PREFILL, COMBINE, EVICT = range(6)
_lib = None


def lib() -> ctypes.CDLL:
    global _lib
    if _lib is None:
        nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
        cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
        if not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
            cuda = "/usr/local/cuda/include"
        os.makedirs(build.OUT, exist_ok=True)
        out = os.path.join(build.OUT, f"libsq_fake.{os.getpid()}.so")
        subprocess.run(
            ["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden", "-Bsymbolic",
             "-I" + cuda, "-I" + build.INCLUDE, "-o", out, os.path.join(HERE, "fake_device.cpp"),
             os.path.join(build.CSRC, "api", "sq_api.cpp"),
             os.path.join(build.CSRC, "host", "core.cpp"), "-ldl"], check=True)
        L = ctypes.CDLL(out)
        os.remove(out)
        for name, (res, args) in _SIGS.items():
            f = getattr(L, name)
            f.restype, f.argtypes = res, args
        L.fake_count.restype = L.fake_races.restype = ctypes.c_int64
        L.fake_malloc_limit.argtypes = [ctypes.c_int64]
        _lib = L
    return _lib
