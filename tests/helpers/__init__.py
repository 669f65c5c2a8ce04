"""Helpers that only tests use."""
import ctypes as C
import os
import shutil
import subprocess
import tempfile

_HERE = os.path.dirname(os.path.abspath(__file__))
_SRC = os.path.join(_HERE, "early_producer.cu")
_LIB = os.path.join(_HERE, "libearly_producer.so")


def early_producer_lib():
    """The producer kernel of early_producer.cu, compiled for sm_100a next to its source."""
    if not os.path.exists(_LIB) or os.path.getmtime(_LIB) < os.path.getmtime(_SRC):
        tmp = _LIB + f".{os.getpid()}.tmp"
        subprocess.check_call(["nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-O2", "-shared",
                               "-Xcompiler", "-fPIC", "-o", tmp, _SRC])
        os.replace(tmp, _LIB)
    L = C.CDLL(_LIB)
    L.early_producer.restype = C.c_int
    L.early_producer.argtypes = [C.c_void_p, C.c_void_p, C.c_size_t, C.c_longlong, C.c_void_p]
    return L


_FAKE = os.path.join(_HERE, "libomnidraft_fake.so")


def fake_runtime_lib():
    """The library's host code on the CUDA runtime of fake_cudart.cu, which runs nothing and writes down the launches."""
    from paper_2507_02659_b200 import build
    src = os.path.join(_HERE, "fake_cudart.cu")
    if not os.path.exists(_FAKE) or os.path.getmtime(_FAKE) < max(build._newest_source(), os.path.getmtime(src)):
        with tempfile.TemporaryDirectory() as tmp:
            nvcc, jobs, objects = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), [], []
            for path in [os.path.join(build.CSRC, f) for f in build.SOURCES] + [src]:
                objects.append(os.path.join(tmp, os.path.basename(path) + ".o"))
                # (host code only: the device code is parsed and not compiled)
                jobs.append(subprocess.Popen([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-Xcompiler", "-fPIC",
                                              "--fdevice-syntax-only", "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC,
                                              "-c", "-o", objects[-1], path]))
            assert [j.wait() for j in jobs] == [0] * len(jobs)
            lib = os.path.join(tmp, "fake.so")
            # -Bsymbolic: torch has the real runtime in the process
            subprocess.check_call(["g++", "-shared", "-Wl,-Bsymbolic", "-Wl,-z,defs", "-o", lib] + objects)
            shutil.move(lib, _FAKE + f".{os.getpid()}.tmp")
        os.replace(_FAKE + f".{os.getpid()}.tmp", _FAKE)
    L = C.CDLL(_FAKE)
    L.fake_log.restype = C.c_char_p
    L.fake_pin.argtypes = [C.c_void_p, C.c_size_t]
    return L
