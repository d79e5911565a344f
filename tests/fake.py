"""The host side of the library on a fake device (fake_device.cpp), for tests that need no GPU."""
import ctypes
import os
import subprocess

from paper_2604_13407_gb300 import build as B
from paper_2604_13407_gb300 import lbm

HERE = os.path.dirname(os.path.abspath(__file__))


def load(folder):
    """Links the host objects with the fake device into folder/libfake.so and loads it in the library's place."""
    B.build()
    out = os.path.join(str(folder), "libfake.so")
    cuda = os.path.dirname(os.path.dirname(subprocess.run(["sh", "-c", "command -v nvcc"], capture_output=True, text=True).stdout.strip()))
    objs = [os.path.join(B.OUT, o) for o in ("lbm_api.o", "lbm_adjoint.o", "lbm_lbana.o")]
    if not all(os.path.exists(o) for o in objs):
        B.build(force=True)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-fvisibility=hidden", "-Wl,-Bsymbolic", "-I", os.path.join(cuda or "/usr/local/cuda", "include"), os.path.join(HERE, "fake_device.cpp")] + objs + ["-o", out], check=True)
    lib = lbm.load_library(out)
    lib.fake_limit.argtypes = [ctypes.c_long, ctypes.c_size_t]
    lib.fake_reset.restype = lib.fake_limit.restype = None
    lib.fake_faults.restype = lib.fake_launches.restype = lib.fake_small_asked.restype = lib.fake_mallocs.restype = lib.fake_attributes.restype = ctypes.c_long
    lib.fake_what.restype = lib.fake_last_step.restype = ctypes.c_char_p
    lib.fake_bytes.restype = ctypes.c_size_t
    return lib


def limit(lib, mallocs=-1, nbytes=-1):
    """The next `mallocs` allocations, of `nbytes` in all, succeed (-1: any)."""
    lib.fake_limit(mallocs, ctypes.c_size_t(nbytes).value)


def sound(lib):
    assert lib.fake_faults() == 0, lib.fake_what().decode()
