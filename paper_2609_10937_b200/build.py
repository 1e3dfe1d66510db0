"""Builds libattn_b200.so (nvcc, sm_100a only) and _fast (g++, the usual calls of binding.py) next to this file.

The library needs CUDA's compiler and headers only.  _fast needs torch's and Python's headers as well, and the versions it was compiled
against, which its file name carries; without it binding.py makes every call itself.
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
import warnings
from importlib import metadata
from pathlib import Path

PKG = Path(__file__).resolve().parent
ROOT = PKG.parent
CSRC = PKG / "csrc"
LIB = PKG / "libattn_b200.so"
SOURCES = [CSRC / "attn_api.cu", CSRC / "attn_plan.cpp"]
HEADERS = [CSRC / "attn_kernels.cuh", CSRC / "decode_kernels.cuh", CSRC / "pipe_kernel.cuh", CSRC / "narrow_kernel.cuh", CSRC / "kv_ring.h", CSRC / "gemm_kernels.cuh", CSRC / "ptx_sm100.cuh", CSRC / "attn_plan_internal.h",
           ROOT / "include" / "attn.h", ROOT / "include" / "gemm.h"]
FAST_SOURCES = [CSRC / "py_fast.cpp", ROOT / "include" / "attn.h", ROOT / "include" / "gemm.h"]


def _stale(out: Path, sources) -> bool:
    return not out.exists() or any(p.stat().st_mtime > out.stat().st_mtime for p in sources)


def fast_path() -> Path:
    """Where the module for this interpreter and this torch is."""
    try:
        torch = metadata.version("torch")
    except metadata.PackageNotFoundError:
        torch = "none"
    return PKG / f"_fast.{sysconfig.get_config_var('SOABI')}.torch-{torch}.so"


def needs_build() -> bool:
    return _stale(LIB, SOURCES + HEADERS) or _stale(fast_path(), FAST_SOURCES)


def _fast_command(out: Path) -> list:
    import torch

    lib = Path(torch.__file__).parent / "lib"
    include = Path(torch.__file__).parent / "include"
    cuda = Path(os.environ.get("CUDA_HOME", "/usr/local/cuda")) / "include"
    return ([os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
            + [f"-I{p}" for p in (ROOT / "include", include, include / "torch" / "csrc" / "api" / "include", cuda, sysconfig.get_paths()["include"])]
            + ["-o", str(out), str(CSRC / "py_fast.cpp"), f"-L{lib}", f"-Wl,-rpath,{lib}", "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"])


def _build_fast() -> None:
    out = fast_path()
    tmp = out.with_name(f"{out.name}.tmp{os.getpid()}")
    try:
        subprocess.run(_fast_command(tmp), check=True)
        os.replace(tmp, out)
    except (ImportError, OSError, subprocess.CalledProcessError) as e:
        for left in (tmp, out):                               # (what is there is of older sources)
            left.unlink(missing_ok=True)
        warnings.warn(f"{out.name} was not built ({e}): binding.py makes every call itself")
    for old in PKG.glob("_fast*.so"):                         # of other versions
        if old != out:
            old.unlink(missing_ok=True)


def build(force: bool = False, verbose: bool = False) -> Path:
    _build_lib(force, verbose)
    if force or _stale(fast_path(), FAST_SOURCES):
        _build_fast()
    return LIB


def _build_lib(force: bool, verbose: bool) -> None:
    if not force and not _stale(LIB, SOURCES + HEADERS):
        return
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB.with_suffix(f".so.tmp{os.getpid()}")
    cmd = [nvcc, "-std=c++17", "-O3", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
           "-Xcompiler", "-fPIC", "-shared", "-I", str(ROOT / "include"), "-I", str(CSRC),
           "-o", str(tmp)] + [str(s) for s in SOURCES]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    subprocess.run(cmd, check=True)
    os.replace(tmp, LIB)


if __name__ == "__main__":
    build(force=True, verbose="-v" in sys.argv)
    print(LIB)
