"""The library's host half (csrc/api.cpp) over a stand-in for the CUDA runtime and the kernel
launchers (cuda_stand_in.cpp): planning, uploads and launch decisions without a GPU."""
import ctypes
import os
import subprocess

import numpy as np

from paper_2602_05017_gb300 import binding
from paper_2602_05017_gb300 import build as libbuild

HERE = os.path.dirname(os.path.abspath(__file__))
RTLD_LAZY = 1


class PipeLaunch(ctypes.Structure):
    _fields_ = [(f, ctypes.c_int) for f in ("mode", "cw", "maxm", "grid", "overlap")]


def load(folder):
    """Compile into `folder` and load; bound lazily, for the launchers no test reaches."""
    so = os.path.join(folder, "libhost.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(libbuild.nvcc())), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-z,lazy,-Bsymbolic", "-I", cuda,
                    "-I", os.path.join(libbuild.ROOT, "include"), "-I", libbuild.CSRC, "-o", so,
                    os.path.join(libbuild.CSRC, "api.cpp"), os.path.join(HERE, "cuda_stand_in.cpp")],
                   check=True)
    dl = ctypes.CDLL(None)
    dl.dlopen.restype = ctypes.c_void_p
    dl.dlopen.argtypes = [ctypes.c_char_p, ctypes.c_int]
    handle = dl.dlopen(so.encode(), RTLD_LAZY)
    assert handle, so
    lib = ctypes.CDLL(so, handle=handle)
    vp, dp = ctypes.c_void_p, ctypes.POINTER(ctypes.c_double)
    lib.biofvm_create.argtypes = [ctypes.POINTER(binding.Grid), ctypes.c_double, ctypes.c_double,
                                  dp, dp, vp, ctypes.c_int, ctypes.c_size_t, ctypes.POINTER(vp)]
    lib.biofvm_batch_create.argtypes = [ctypes.c_int, ctypes.POINTER(binding.Grid), dp, dp, dp, dp,
                                        ctypes.c_int, ctypes.c_size_t, vp, ctypes.POINTER(vp)]
    lib.biofvm_describe.argtypes = [vp, ctypes.c_char_p, ctypes.c_size_t]
    lib.biofvm_step.argtypes = [vp, ctypes.c_int]
    lib.biofvm_step_save.argtypes = [vp, vp]
    lib.biofvm_adjoint_step.argtypes = [vp] * 7
    lib.biofvm_set_sources.argtypes = [vp, ctypes.c_int64] + [vp] * 5
    lib.biofvm_destroy.argtypes = [vp]
    lib.biofvm_batch_env.argtypes = [vp, ctypes.c_int, ctypes.POINTER(vp)]
    lib.biofvm_batch_step.argtypes = [vp, ctypes.c_int]
    lib.biofvm_batch_destroy.argtypes = [vp]
    lib.stand_in_fail_allocation.argtypes = [ctypes.c_long]
    return lib


def _params(ns):
    a = np.full(ns, 1e3), np.full(ns, 0.1)
    return a, [v.ctypes.data_as(ctypes.POINTER(ctypes.c_double)) for v in a]


def create(lib, nx, ny, nz, ns, precision):
    """(status, handle)"""
    keep, (D, lam) = _params(ns)
    h = ctypes.c_void_p()
    st = lib.biofvm_create(ctypes.byref(binding.Grid(nx, ny, nz, ns)), 20.0, 0.01, D, lam, None,
                           binding.PRECISIONS[precision], 0, ctypes.byref(h))
    return st, h


def create_batch(lib, grids, precision):
    n = len(grids)
    keep, (D, lam) = _params(sum(g[3] for g in grids))
    h3 = np.full(n, 20.0), np.full(n, 0.01)
    dx, dt = (v.ctypes.data_as(ctypes.POINTER(ctypes.c_double)) for v in h3)
    b = ctypes.c_void_p()
    st = lib.biofvm_batch_create(n, (binding.Grid * n)(*[binding.Grid(*g) for g in grids]), dx, dt,
                                 D, lam, binding.PRECISIONS[precision], 0, None, ctypes.byref(b))
    return st, b


def describe(lib, h):
    out = ctypes.create_string_buffer(256)
    assert lib.biofvm_describe(h, out, 256) == binding.OK
    return out.value.decode()


def pipe_launches(lib):
    out = (PipeLaunch * 4096)()
    n = lib.stand_in_pipe_launches(out, 4096)
    return [out[i] for i in range(min(n, 4096))]


def last_error(lib):
    lib.biofvm_last_error.restype = ctypes.c_char_p
    return lib.biofvm_last_error().decode()
