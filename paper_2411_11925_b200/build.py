"""Builds libcsd.so (the C-ABI CUDA library, nvcc for sm_100a) and _marshal (argument marshalling of its short calls) in-tree."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "libcsd.so")
MARSHAL_PATH = os.path.join(PKG_DIR, "_marshal" + sysconfig.get_config_var("EXT_SUFFIX"))
ABI_HEADER = os.path.join(os.path.dirname(PKG_DIR), "include", "csd.h")
SOURCES = ["csd_api.cu"]
HEADERS = ["ptx.cuh", "epilogue.cuh", "gemm.cuh", "rowops.cuh", "fold.cuh", "groupchain.cuh", "wideplan.h", "widechain.cuh", "gmm.cuh", "f32chain.cuh"]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _stale(target: str, sources) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(s) > os.path.getmtime(target) for s in sources)


def needs_build() -> bool:
    return _stale(LIB_PATH, [os.path.join(CSRC, f) for f in SOURCES + HEADERS] + [ABI_HEADER])


def _run(cmd) -> subprocess.CompletedProcess:
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("build failed:\n" + " ".join(cmd) + "\n" + res.stdout + res.stderr)
    return res


def build_library(force: bool = False, verbose: bool = False) -> str:
    if force or needs_build():
        res = _run([_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
                    "-shared", "-Xcompiler", "-fPIC", "-cudart", "static", "-Xptxas", "-v" if verbose else "-O3",
                    "-Xlinker", "-soname=libcsd.so", "-o", LIB_PATH] + [os.path.join(CSRC, s) for s in SOURCES])
        if verbose:
            print(res.stderr)
    build_marshal(force)
    return LIB_PATH


def build_marshal(force: bool = False) -> str:
    src = os.path.join(CSRC, "marshal.cpp")
    if force or _stale(MARSHAL_PATH, [src, ABI_HEADER]):
        import torch
        from torch.utils import cpp_extension
        libs = os.path.join(os.path.dirname(torch.__file__), "lib")
        inc = [f"-I{d}" for d in cpp_extension.include_paths() + [sysconfig.get_paths()["include"]]]
        _run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"] + inc
             + [src, "-o", MARSHAL_PATH, f"-L{PKG_DIR}", "-l:libcsd.so", f"-L{libs}", "-ltorch_python", "-ltorch_cpu", "-lc10",
                "-Wl,-rpath,$ORIGIN", f"-Wl,-rpath,{libs}"])
    return MARSHAL_PATH


if __name__ == "__main__":
    print(build_library(force=True, verbose="-v" in sys.argv))
