"""Builds libomnidraft.so (the C-ABI CUDA library, nvcc for sm_100a) and _marshal.so (the
binding's argument marshalling, a Python extension) in-tree."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libomnidraft.so")
EXT = os.path.join(HERE, "_marshal.so")
EXT_FOR = os.path.join(HERE, "_build", "marshal_built_for")
SOURCES = ["od_api.cu", "od_map.cu", "od_verify.cu", "od_sample.cu", "od_step.cu", "od_host.cu", "od_noalloc.cu", "od_exit.cu", "od_cache.cu", "od_distill.cu"]


def _newest_source() -> float:
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    files.append(os.path.join(ROOT, "include", "omnidraft.h"))
    return max(os.path.getmtime(f) for f in files)


def build(force: bool = False, verbose: bool = False) -> str:
    _build_lib(force, verbose)
    _build_marshal(force, verbose)
    return LIB


def built_for() -> str:
    """What _marshal.so depends on besides its sources."""
    import platform
    import torch
    return f"python {platform.python_version()}, torch {torch.__version__}"


def _build_marshal(force: bool = False, verbose: bool = False) -> None:
    """The extension is optional: without it (no g++, no torch headers) the binding marshals in Python."""
    import sysconfig
    import torch
    fresh = os.path.exists(EXT) and os.path.getmtime(EXT) >= _newest_source()
    if not force and fresh and os.path.exists(EXT_FOR) and open(EXT_FOR).read() == built_for():
        return
    root = os.path.dirname(torch.__file__)
    inc = os.path.join(root, "include")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    tmp = EXT + f".{os.getpid()}.tmp"
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
           f'-DOD_BUILT_FOR="{built_for()}"',
           "-I", os.path.join(ROOT, "include"), "-I", inc, "-I", os.path.join(inc, "torch", "csrc", "api", "include"),
           "-I", os.path.join(cuda, "include"), "-I", sysconfig.get_paths()["include"], "-o", tmp,
           os.path.join(CSRC, "marshal.cpp"), "-L", HERE, "-l:libomnidraft.so", "-L", os.path.join(root, "lib"),
           "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda",
           "-Wl,-rpath,$ORIGIN:" + os.path.join(root, "lib")]
    try:
        res = subprocess.run(cmd, capture_output=True, text=True)
        failed, said = res.returncode != 0, res.stdout + res.stderr
    except OSError as e:
        failed, said = True, f"{e}\n"
    if verbose or failed:
        sys.stderr.write(said)
    if failed:
        sys.stderr.write("_marshal.so could not be built: the binding will look at its arguments in Python\n")
        if os.path.exists(EXT):                             # of other sources, or for another torch
            os.remove(EXT)
        return
    os.replace(tmp, EXT)
    os.makedirs(os.path.dirname(EXT_FOR), exist_ok=True)
    with open(EXT_FOR, "w") as f:
        f.write(built_for())


def _build_lib(force: bool = False, verbose: bool = False) -> str:
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _newest_source():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + f".{os.getpid()}.tmp"
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3",
           "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-Xlinker", "-soname=libomnidraft.so", "-Xptxas", "-v",
           "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", tmp]
    cmd += [os.path.join(CSRC, s) for s in SOURCES]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed building libomnidraft.so")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
