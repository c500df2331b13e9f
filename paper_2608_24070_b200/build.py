"""Build in-tree: ``libslope.so`` (the C-ABI CUDA library, nvcc for sm_100a) and ``_slope.so`` (the binding's native
argument marshalling, g++ against torch's headers)."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig
from pathlib import Path

PKG = Path(__file__).resolve().parent
CSRC = PKG / "csrc"
LIB = PKG / "libslope.so"
SOURCES = [CSRC / "slope_lib.cu"]
HEADERS = sorted(CSRC.glob("*.cuh")) + [PKG.parent / "include" / "slope.h"]
NATIVE = PKG / "_slope.so"
NATIVE_SOURCES = [CSRC / "py_binding.cpp", PKG.parent / "include" / "slope.h"]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-lineinfo", "-std=c++17",
    "-shared", "-Xcompiler", "-fPIC",
]


def nvcc_path() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found; cannot build libslope.so")


def _newer(target: Path, sources) -> bool:
    if not target.exists():
        return False
    t = target.stat().st_mtime
    return all(p.stat().st_mtime <= t for p in sources)


def native_build() -> str:
    """What _slope.so depends on besides its sources: torch's C++ interface and this interpreter's."""
    import torch

    return (f"_slope.so for torch {torch.__version__}, C++11 ABI {int(torch._C._GLIBCXX_USE_CXX11_ABI)}, "
            f"{sysconfig.get_config_var('SOABI')}")


def native_matches() -> bool:
    """_slope.so is there and was compiled against this torch and this Python (it carries native_build() as a string)."""
    return NATIVE.exists() and native_build().encode() + b"\0" in NATIVE.read_bytes()


def _native_current() -> bool:
    return _newer(NATIVE, NATIVE_SOURCES) and native_matches()


def up_to_date() -> bool:
    return _newer(LIB, SOURCES + HEADERS) and _native_current()


def _compile(cmd, target: Path) -> None:
    tmp = target.with_suffix(f".{os.getpid()}.tmp")
    subprocess.check_call([*cmd, "-o", str(tmp)])
    os.replace(tmp, target)


def native_command():
    import torch

    root = Path(torch.__file__).resolve().parent
    cuda = Path(nvcc_path()).resolve().parent.parent
    abi = int(torch._C._GLIBCXX_USE_CXX11_ABI)
    return ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={abi}",
            f'-DSLOPE_NATIVE_BUILD="{native_build()}"',
            f"-I{root / 'include'}", f"-I{sysconfig.get_paths()['include']}", f"-I{cuda / 'include'}",
            str(NATIVE_SOURCES[0]), f"-L{root / 'lib'}", "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]


def build(force: bool = False, verbose: bool = False) -> Path:
    if force or not _newer(LIB, SOURCES + HEADERS):
        _compile([nvcc_path(), *NVCC_FLAGS, *(["-Xptxas", "-v"] if verbose else []), *map(str, SOURCES)], LIB)
    if force or not _native_current():
        _compile(native_command(), NATIVE)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
