"""Builds libqamw.so (CUDA kernels + C ABI) in-tree with nvcc for sm_100a, and _qamw.so, its Python entry, with g++."""
from __future__ import annotations

import os
import subprocess
import sysconfig

_PKG = os.path.dirname(os.path.abspath(__file__))
_CSRC = os.path.join(_PKG, "csrc")
_INC = os.path.join(os.path.dirname(_PKG), "include")
LIB_PATH = os.path.join(_PKG, "libqamw.so")
EXT_PATH = os.path.join(_PKG, "_qamw.so")
EXT_SOURCE = "qamw_py.cpp"
SOURCES = ["qamw_kernels.cu", "qamw_rows.cu", "qamw_prepare.cu", "qamw_lloyd.cu", "qamw_variants.cu", "qamw_gemv.cu", "qamw_host.cpp", "qamw_table.cpp"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC,-Wall,-Wextra", "-shared", "-t", "0"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def _stale(path: str, deps) -> bool:
    return not os.path.exists(path) or any(os.path.getmtime(d) > os.path.getmtime(path) for d in deps)


def _lib_deps():
    return [os.path.join(_CSRC, f) for f in os.listdir(_CSRC) if f != EXT_SOURCE] + [os.path.join(_INC, "qamw.h")]


def _ext_deps():
    return [os.path.join(_CSRC, EXT_SOURCE), os.path.join(_INC, "qamw.h")]


def needs_build() -> bool:
    return _stale(LIB_PATH, _lib_deps()) or _stale(EXT_PATH, _ext_deps())


def _build_ext():
    import torch
    from torch.utils import cpp_extension

    libs = os.path.join(os.path.dirname(torch.__file__), "lib")
    cuda = os.path.dirname(os.path.dirname(_nvcc())) if os.path.isabs(_nvcc()) else "/usr/local/cuda"
    tmp = EXT_PATH + f".tmp{os.getpid()}"
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-o", tmp, os.path.join(_CSRC, EXT_SOURCE), "-I", _INC,
           "-I", sysconfig.get_paths()["include"], "-I", os.path.join(cuda, "include")]
    cmd += [x for d in cpp_extension.include_paths() for x in ("-isystem", d)]
    cmd += ["-L", _PKG, "-l:libqamw.so", "-Wl,-rpath,$ORIGIN", "-L", libs, "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda",
            f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    subprocess.run(cmd, check=True)
    os.replace(tmp, EXT_PATH)


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _stale(LIB_PATH, _lib_deps()):
        tmp = LIB_PATH + f".tmp{os.getpid()}"
        cmd = [_nvcc(), *NVCC_FLAGS, "-I", _INC, "-I", _CSRC, "-o", tmp, "-Xlinker", "-soname=libqamw.so"]
        if verbose:
            cmd += ["-Xptxas", "-v"]
        cmd += [os.path.join(_CSRC, s) for s in SOURCES]
        subprocess.run(cmd, check=True)
        os.replace(tmp, LIB_PATH)
    if force or _stale(EXT_PATH, _ext_deps()):
        _build_ext()
    return LIB_PATH


if __name__ == "__main__":
    import sys
    print(build(force=True, verbose="-v" in sys.argv))
