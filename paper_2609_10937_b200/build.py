"""Builds libattn_b200.so (nvcc, sm_100a only) and _fast.so (g++, the usual calls of binding.py) next to this file."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from pathlib import Path

PKG = Path(__file__).resolve().parent
ROOT = PKG.parent
CSRC = PKG / "csrc"
LIB = PKG / "libattn_b200.so"
FAST = PKG / "_fast.so"
SOURCES = [CSRC / "attn_api.cu", CSRC / "attn_plan.cpp"]
HEADERS = [CSRC / "attn_kernels.cuh", CSRC / "decode_kernels.cuh", CSRC / "pipe_kernel.cuh", CSRC / "narrow_kernel.cuh", CSRC / "kv_ring.h", CSRC / "gemm_kernels.cuh", CSRC / "ptx_sm100.cuh", CSRC / "attn_plan_internal.h",
           ROOT / "include" / "attn.h", ROOT / "include" / "gemm.h"]
FAST_SOURCES = [CSRC / "py_fast.cpp", ROOT / "include" / "attn.h", ROOT / "include" / "gemm.h"]


def _stale(out: Path, sources) -> bool:
    return not out.exists() or any(p.stat().st_mtime > out.stat().st_mtime for p in sources)


def needs_build() -> bool:
    return _stale(LIB, SOURCES + HEADERS) or _stale(FAST, FAST_SOURCES)


def _fast_command(out: Path) -> list:
    import torch

    lib = Path(torch.__file__).parent / "lib"
    include = Path(torch.__file__).parent / "include"
    cuda = Path(os.environ.get("CUDA_HOME", "/usr/local/cuda")) / "include"
    return ([os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
            + [f"-I{p}" for p in (ROOT / "include", include, include / "torch" / "csrc" / "api" / "include", cuda, sysconfig.get_paths()["include"])]
            + ["-o", str(out), str(CSRC / "py_fast.cpp"), f"-L{lib}", f"-Wl,-rpath,{lib}", "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"])


def build(force: bool = False, verbose: bool = False) -> Path:
    if force or _stale(FAST, FAST_SOURCES):
        tmp = FAST.with_suffix(f".so.tmp{os.getpid()}")
        subprocess.run(_fast_command(tmp), check=True)
        os.replace(tmp, FAST)
    if not force and not _stale(LIB, SOURCES + HEADERS):
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB.with_suffix(f".so.tmp{os.getpid()}")
    cmd = [nvcc, "-std=c++17", "-O3", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
           "-Xcompiler", "-fPIC", "-shared", "-I", str(ROOT / "include"), "-I", str(CSRC),
           "-o", str(tmp)] + [str(s) for s in SOURCES]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    subprocess.run(cmd, check=True)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    build(force=True, verbose="-v" in sys.argv)
    print(LIB)
