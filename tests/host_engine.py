"""The library's objects linked against tests/fake_cuda/runtime.cpp in place of the CUDA runtime: contexts,
plans and requests on the CPU, for tests of the engine's host side (kernels are counted, not run)."""
import ctypes
import os
import subprocess

from paper_0906_5170_gb300 import build as pkbuild
from paper_0906_5170_gb300 import capi

SRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fake_cuda", "runtime.cpp")


def build():
    pkbuild.build()
    objs = [os.path.join(pkbuild.OUT_DIR, f + ".o") for f in pkbuild.CU + pkbuild.CXX]
    if not all(os.path.exists(o) for o in objs):
        pkbuild.build(force=True)
    lib = os.path.join(pkbuild.OUT_DIR, "libcasimir_host.so")
    tmp = lib + f".{os.getpid()}.tmp"
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I", pkbuild.CSRC,
                           "-I", os.path.join(pkbuild.ROOT, "include"), "-I", "/usr/local/cuda/include", "-o", tmp,
                           SRC, *objs, "-lpthread"])
    os.replace(tmp, lib)
    return lib


def load(path):
    """Make the fake-runtime library the one the package calls; returns it (with the fake_* functions)."""
    L = ctypes.CDLL(path)
    for name, (res, args) in capi.SIGNATURES.items():
        f = getattr(L, name)
        f.restype = res
        f.argtypes = args
    for name in ("fake_launches", "fake_queries", "fake_captures", "fake_host_frees"):
        getattr(L, name).restype = ctypes.c_int64
    L.fake_launches.argtypes = [ctypes.c_char_p]
    L.fake_cost.argtypes = [ctypes.c_char_p, ctypes.c_double]
    L.fake_cost.restype = None
    capi._lib = L
    return L
