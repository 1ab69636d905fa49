"""Builds libvector.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and the extension module that marshals arguments."""
from __future__ import annotations

import os
import subprocess
import sys
import warnings

from .binding import marshal_path

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
LIB = os.path.join(HERE, "libvector.so")

SOURCES = ["host.cpp", "score.cu", "keydiff.cu", "route.cu", "compact.cu", "decode.cu", "decode_layer.cu", "diagnostics.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xptxas=-v",
              "-Xcompiler", "-fPIC,-O3,-fvisibility=hidden", "-I", INCLUDE, "-I", CSRC]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    raise RuntimeError("nvcc not found")


def _older(target: str, deps) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in [*deps, os.path.join(INCLUDE, "vector.h"), __file__])


def _stale() -> bool:
    return _older(LIB, [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f != "marshal.cpp"])


def build_marshal(force: bool = False) -> str:
    """The extension module behind the binding (csrc/marshal.cpp): plain C++ against the headers of Python and torch."""
    src, target = os.path.join(CSRC, "marshal.cpp"), marshal_path()
    if not force and not _older(target, [src]):
        return target
    import shutil
    import sysconfig
    import torch
    from torch.utils.cpp_extension import include_paths, library_paths
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(shutil.which(_nvcc()) or _nvcc())))
    incs = [INCLUDE, *include_paths(), sysconfig.get_paths()["include"], os.path.join(cuda, "include")]
    tmp = target + f".tmp{os.getpid()}"
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
                           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}", *(f"-I{i}" for i in incs), src,
                           *(f"-L{p}" for p in library_paths()), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-o", tmp])
    os.replace(tmp, target)
    return target


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every translation unit to an object and link the shared library.  Extra nvcc flags can be
    given in the environment variable VECTOR_NVCC_FLAGS (e.g. -DVECTOR_SCORE_POLY16=6 for the sweep of the
    share of softmax exponentials evaluated on the FMA pipe).  The library comes first and needs nvcc only; where the extension module
    cannot be compiled, that is a warning."""
    if force or _stale():
        _build_library(verbose)
    try:
        build_marshal(force)
    except Exception as e:
        warnings.warn(f"the extension module that marshals arguments was not built ({e!r}): it needs a C++ compiler, Python's headers and a CUDA build of "
                      "torch; without it every call goes through ctypes", RuntimeWarning)
    return LIB


def _build_library(verbose: bool) -> None:
    objdir = os.path.join(HERE, "_build")
    os.makedirs(objdir, exist_ok=True)
    nvcc = _nvcc()
    procs = []
    for src in SOURCES:
        obj = os.path.join(objdir, src + ".o")
        cmd = [nvcc, *NVCC_FLAGS, *os.environ.get("VECTOR_NVCC_FLAGS", "").split(), "-c", os.path.join(CSRC, src), "-o", obj]
        procs.append((src, obj, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    objs = []
    for src, obj, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode != 0:
            sys.stderr.write(out)
        if p.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}")
        with open(os.path.join(objdir, src + ".ptxas.txt"), "w") as f:
            f.write(out)
        objs.append(obj)
    tmp = LIB + f".tmp{os.getpid()}"
    subprocess.check_call([nvcc, "-shared", "-o", tmp, *objs, "-gencode", "arch=compute_100a,code=sm_100a"])
    os.replace(tmp, LIB)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
