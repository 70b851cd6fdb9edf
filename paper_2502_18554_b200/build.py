"""Builds libzccl.so (the C-ABI library, nvcc for sm_100a) and _zccl.so (its CPython module) in-tree."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from pathlib import Path

PKG = Path(__file__).resolve().parent
CSRC = PKG / "csrc"
LIB = PKG / "libzccl.so"
MODULE = PKG / "_zccl.so"
MODULE_SOURCE = CSRC / "zccl_binding.cpp"
SOURCES = [CSRC / "zccl_kernels.cu", CSRC / "zccl_codec.cu", CSRC / "zccl_api.cu", CSRC / "zccl_noalloc.cu", CSRC / "zccl_generic.cu"]
HEADERS = [CSRC / "zccl_internal.h", CSRC / "zccl_device.cuh", CSRC / "zccl_tiles.cuh", CSRC / "zccl_decode.cuh", CSRC / "zccl_stream.cuh", CSRC / "zccl_hop.cuh", CSRC / "zccl_ring.cuh", CSRC / "zccl_codec_f64.cuh", CSRC / "zccl_codec_tiled.cuh", PKG.parent / "include" / "zccl.h"]

NVCC_FLAGS = [
    "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
    "--fmad=false",                       # no contraction anywhere: streams must be reproducible bit for bit
    "-Xcompiler", "-fPIC,-ffp-contract=off,-fno-fast-math",
    "-shared", "-cudart", "shared",
]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (cand == "nvcc" or Path(cand).exists()):
            return cand
    raise RuntimeError("nvcc not found")


def _stale(target: Path, sources) -> bool:
    if not target.exists():
        return True
    t = target.stat().st_mtime
    return any(p.stat().st_mtime > t for p in sources)


def needs_build() -> bool:
    return _stale(LIB, SOURCES + HEADERS)


def build_module(force: bool = False) -> Path:
    """The CPython module, linked against libzccl.so beside it and the installed torch."""
    if not force and not _stale(MODULE, [MODULE_SOURCE, PKG.parent / "include" / "zccl.h"]):
        return MODULE
    import torch
    root = Path(torch.__file__).resolve().parent
    cuda = Path(nvcc()).resolve().parent.parent
    tmp = MODULE.with_suffix(f".tmp{os.getpid()}.so")
    subprocess.check_call(
        ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
         f"-I{sysconfig.get_paths()['include']}", f"-I{root / 'include'}", f"-I{root / 'include/torch/csrc/api/include'}", f"-I{cuda / 'include'}",
         "-o", str(tmp), str(MODULE_SOURCE), f"-L{PKG}", "-l:libzccl.so", "-Wl,-rpath,$ORIGIN", f"-L{root / 'lib'}",
         "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"])
    os.replace(tmp, MODULE)
    return MODULE


def build(force: bool = False, verbose: bool = False, extra: list[str] | None = None) -> Path:
    if force or needs_build():
        tmp = LIB.with_suffix(f".tmp{os.getpid()}.so")
        extra = list(extra or []) + os.environ.get("ZCCL_NVCC_EXTRA", "").split()
        cmd = [nvcc(), *NVCC_FLAGS, *extra, "-o", str(tmp), *map(str, SOURCES)]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
            print(" ".join(cmd), file=sys.stderr)
        subprocess.check_call(cmd)
        os.replace(tmp, LIB)
    build_module(force)
    return LIB


if __name__ == "__main__":
    build(force=True, verbose="-v" in sys.argv)
    print(LIB)
