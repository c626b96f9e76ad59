"""Compile the CUDA library in-tree for sm_100a (nvcc cross-compiles without a GPU)."""
from __future__ import annotations

import os
import subprocess
import sys
from pathlib import Path

PKG = Path(__file__).resolve().parent
ROOT = PKG.parent
SO = PKG / "libsla.so"
SOURCES = sorted((PKG / "csrc").glob("*.cu"))
HEADERS = sorted((PKG / "csrc").glob("*.h")) + sorted((PKG / "csrc").glob("*.cuh")) + [ROOT / "include" / "sla.h"]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-shared", f"-I{ROOT / 'include'}", f"-I{PKG / 'csrc'}",
]


def build(force: bool = False, verbose: bool = False) -> Path:
    newest = max(p.stat().st_mtime for p in SOURCES + HEADERS)
    if not force and SO.exists() and SO.stat().st_mtime >= newest:
        return SO
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = SO.with_suffix(f".so.{os.getpid()}.tmp")
    cmd = [nvcc, *NVCC_FLAGS, *(["-Xptxas", "-v"] if verbose else []), "-o", str(tmp), *map(str, SOURCES)]
    subprocess.run(cmd, check=True)
    os.replace(tmp, SO)
    return SO


FAST_SO = PKG / "_sla_fast.so"
FAST_SOURCE = PKG / "native" / "fastcall.cpp"


def build_fast(force: bool = False) -> Path:
    """The native argument marshalling of the decode calls (a Python extension against torch's headers)."""
    if not force and FAST_SO.exists() and FAST_SO.stat().st_mtime >= FAST_SOURCE.stat().st_mtime:
        return FAST_SO
    import sysconfig
    import torch
    t = Path(torch.__file__).resolve().parent
    tmp = FAST_SO.with_suffix(f".so.{os.getpid()}.tmp")
    subprocess.run(["g++", "-O2", "-std=c++20", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
                    f"-I{sysconfig.get_paths()['include']}", f"-I{t / 'include'}", f"-I{t / 'include/torch/csrc/api/include'}",
                    "-I/usr/local/cuda/include", str(FAST_SOURCE), "-o", str(tmp), f"-L{t / 'lib'}", f"-Wl,-rpath,{t / 'lib'}",
                    "-ltorch_python", "-ltorch_cpu", "-ltorch_cuda", "-lc10_cuda", "-lc10"], check=True)
    os.replace(tmp, FAST_SO)
    return FAST_SO


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
    print(build_fast(force="--force" in sys.argv))
