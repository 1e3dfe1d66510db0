"""Builds libattn_b200.so (sm_100a only) next to this file with nvcc."""
from __future__ import annotations

import os
import subprocess
import sys
from pathlib import Path

PKG = Path(__file__).resolve().parent
ROOT = PKG.parent
CSRC = PKG / "csrc"
LIB = PKG / "libattn_b200.so"
SOURCES = [CSRC / "attn_api.cu", CSRC / "attn_plan.cpp"]
HEADERS = [CSRC / "attn_kernels.cuh", CSRC / "decode_kernels.cuh", CSRC / "pipe_kernel.cuh", CSRC / "narrow_kernel.cuh", CSRC / "kv_ring.h", CSRC / "gemm_kernels.cuh", CSRC / "ptx_sm100.cuh", CSRC / "attn_plan_internal.h",
           ROOT / "include" / "attn.h", ROOT / "include" / "gemm.h"]


def needs_build() -> bool:
    if not LIB.exists():
        return True
    t = LIB.stat().st_mtime
    return any(p.stat().st_mtime > t for p in SOURCES + HEADERS)


def build(force: bool = False, verbose: bool = False) -> Path:
    if not force and not needs_build():
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
