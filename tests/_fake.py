"""The library's object files linked with tests/fake_cudart.cpp: the C interface on a CPU, with device
memory in host memory, kernels that do not run, allocations that fail on demand and modelled launch times."""
import ctypes
import glob
import os
import subprocess

from paper_1912_07921_gb300 import _lib, build

HERE = os.path.dirname(os.path.abspath(__file__))
HOOK = ctypes.CFUNCTYPE(ctypes.c_double, ctypes.c_char_p, ctypes.POINTER(ctypes.c_uint), ctypes.POINTER(ctypes.c_uint),
                        ctypes.POINTER(ctypes.c_void_p))


def load(tmp_path):
    """The interface over the fake runtime, a copy of its own (allocations and clock start anew)."""
    build.build()
    so = os.path.join(str(tmp_path), "libtdks_fake.so")
    cuda = os.path.dirname(os.path.dirname(build._nvcc()))
    objs = [os.path.join(build.OUT_DIR, s.replace(".cu", ".o")) for s in build.SOURCES]
    inc = [d for d in [os.path.join(cuda, "include")] + glob.glob(os.path.join(cuda, "targets", "*", "include"))
           if os.path.isdir(d)]
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-Wl,-Bsymbolic", *[f"-I{d}" for d in inc],
                           os.path.join(HERE, "fake_cudart.cpp"), *objs, "-o", so])
    lib = ctypes.CDLL(so)
    for name, (args, res) in _lib.SIGNATURES.items():
        getattr(lib, name).argtypes, getattr(lib, name).restype = args, res
    lib.fake_fail_malloc.argtypes = [ctypes.c_long]
    lib.fake_fail_launch.argtypes = [ctypes.c_long]
    lib.fake_live_blocks.restype = ctypes.c_long
    lib.fake_copies_in_flight.restype = ctypes.c_long
    lib.fake_unordered_launches.restype = ctypes.c_long
    lib.fake_set_hook.argtypes = [HOOK]
    lib.fake_times.argtypes = [ctypes.c_double, ctypes.c_double]
    return lib


def create(lib, nx, ny, nz, h=0.3, order=4, bc=0, prec=0, n_orb=1, n_k=1, stream=None):
    out = ctypes.c_void_p()
    rc = lib.tdks_create_grid(nx, ny, nz, h, order, bc, prec, n_orb, n_k, None, None, stream, ctypes.byref(out))
    assert rc == 0, lib.tdks_last_error()
    return out
