"""csrc/stereo_api.cu built against tests/fake_cuda.cpp, for CPU tests of what the
entry points do on the host: the order of their calls, and what they do when one
of them fails. Nothing here touches a GPU."""
import ctypes
import os
import shutil
import subprocess

from paper_2212_00488_gb300 import _lib

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2212_00488_gb300", "csrc")


def available():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    return os.path.exists(nvcc) and shutil.which("g++") is not None


def build(folder):
    """The fake library in `folder`, with the signatures of the real one."""
    nvcc = os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")
    out = os.path.join(str(folder), "libfake.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-fPIC", "-shared", "-fvisibility=hidden", "-Wl,-Bsymbolic",
                    '-DSTEREO_TEST_API=__attribute__((visibility("default")))', "-I", CSRC,
                    "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include"), "-x", "c++",
                    os.path.join(CSRC, "stereo_api.cu"), os.path.join(HERE, "fake_cuda.cpp"), "-o", out], check=True)
    lib = ctypes.CDLL(out)
    for name, (res, args) in _lib._SIGNATURES.items():
        if hasattr(lib, name):
            fn = getattr(lib, name)
            fn.restype, fn.argtypes = res, args
    lib.fake_log.restype = ctypes.c_char_p
    return lib
