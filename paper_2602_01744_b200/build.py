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


def nvcc_path() -> str:
    return os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


def build(force: bool = False, verbose: bool = False) -> Path:
    newest = max(p.stat().st_mtime for p in SOURCES + HEADERS)
    if not force and SO.exists() and SO.stat().st_mtime >= newest:
        return SO
    nvcc = nvcc_path()
    tmp = SO.with_suffix(f".so.{os.getpid()}.tmp")
    cmd = [nvcc, *NVCC_FLAGS, *(["-Xptxas", "-v"] if verbose else []), "-o", str(tmp), *map(str, SOURCES)]
    subprocess.run(cmd, check=True)
    os.replace(tmp, SO)
    return SO


FAST_SOURCE = PKG / "native" / "fastcall.cpp"


def fast_so() -> Path:
    """Where the extension of this Python, this torch and this source lies.  It is compiled against torch's inline accessors, so one that was built for
    another of the three must not be loaded: all three are in its name."""
    import hashlib
    import sysconfig
    import torch
    key = [sysconfig.get_config_var("SOABI"), torch.__version__, str(int(torch._C._GLIBCXX_USE_CXX11_ABI)), FAST_SOURCE.read_text()]
    return PKG / f"_sla_fast.{hashlib.sha256(chr(0).join(map(str, key)).encode()).hexdigest()[:16]}.so"


def build_fast(force: bool = False) -> Path:
    """The native argument marshalling of the decode calls (a Python extension against torch's headers).  Optional: the binding works without it."""
    so = fast_so()
    if not force and so.exists():
        return so
    import shutil
    import sysconfig
    import torch
    t = Path(torch.__file__).resolve().parent
    cuda = Path(shutil.which(nvcc_path()) or nvcc_path()).resolve().parent.parent         # (the toolkit that compiles the library)
    tmp = so.with_suffix(f".so.{os.getpid()}.tmp")
    subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-std=c++20", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
                    f"-I{sysconfig.get_paths()['include']}", f"-I{t / 'include'}", f"-I{t / 'include/torch/csrc/api/include'}",
                    f"-I{cuda / 'include'}", str(FAST_SOURCE), "-o", str(tmp), f"-L{t / 'lib'}", f"-Wl,-rpath,{t / 'lib'}",
                    "-ltorch_python", "-ltorch_cpu", "-ltorch_cuda", "-lc10_cuda", "-lc10"], check=True)
    os.replace(tmp, so)
    return so


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
    try:
        print(build_fast(force="--force" in sys.argv))
    except Exception as e:
        print(f"decode marshalling not built ({e}): decode calls will take the Python path", file=sys.stderr)
