"""The library's host code over a runtime that runs nothing (fake_cuda.c)."""

import ctypes as C
import functools
import glob
import os
import subprocess
import tempfile

from paper_2607_01757_gb300 import build


@functools.lru_cache(maxsize=None)
def load() -> C.CDLL:
    build.build()
    d = tempfile.mkdtemp(prefix="vt_fake_")
    here = os.path.dirname(os.path.abspath(__file__))
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath("/usr/local/cuda/bin/nvcc"))), "include")
    so, o = os.path.join(d, "libvt_fake.so"), os.path.join(d, "fake_cuda.o")
    subprocess.run(["gcc", "-O1", "-fPIC", "-fvisibility=hidden", "-I", cuda, "-c", os.path.join(here, "fake_cuda.c"),
                    "-o", o], check=True)
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-Wl,-z,defs", "-o", so, o,
                    *sorted(glob.glob(os.path.join(build.OUT_DIR, "*.cu.o")))], check=True)
    return C.CDLL(so)
