"""Build libqbert.so in-tree with nvcc for sm_100a, and the Python entry to it, _qbert, with the host compiler (no
JIT cache: the built libraries travel with the tree)."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from pathlib import Path

from . import EXT_PATH as EXT

PKG = Path(__file__).resolve().parent
CSRC = PKG / "csrc"
INCLUDE = PKG.parent / "include"
LIB = PKG / "libqbert.so"
SOURCES = ["api.cu", "quantize_act.cu", "quantize_weights.cu", "quantize_weights_noalloc.cu", "gemm.cu", "probe.cu", "embedding.cu", "sensitivity.cu"]


def _nvcc() -> str:
    cand = os.environ.get("NVCC") or "/usr/local/cuda/bin/nvcc"
    return cand if Path(cand).exists() else "nvcc"


def _stale(target: Path, *patterns: str) -> bool:
    if not target.exists():
        return True
    t = target.stat().st_mtime
    deps = [d for pattern in patterns for d in CSRC.glob(pattern)] + list(INCLUDE.glob("*.h"))
    return any(d.stat().st_mtime > t for d in deps)


def _lib_stale() -> bool:
    return _stale(LIB, "*.cu", "*.cuh")


def _ext_stale() -> bool:
    return _stale(EXT, "*.cpp")


def needs_build() -> bool:
    return _lib_stale() or _ext_stale()


def _binding_command(out: str) -> list[str]:
    import torch
    root = Path(torch.__file__).resolve().parent
    cuda = Path(_nvcc()).resolve().parent.parent
    return [os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared", "-I", str(INCLUDE),
            "-isystem", str(root / "include"), "-isystem", str(root / "include/torch/csrc/api/include"),
            "-isystem", str(cuda / "include"), "-isystem", sysconfig.get_paths()["include"], str(CSRC / "binding.cpp"), "-o", out,
            "-L", str(root / "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-ltorch_cuda", "-lc10", "-lc10_cuda",
            "-L", str(PKG), "-lqbert", "-Wl,-rpath,$ORIGIN"]


def build(force: bool = False, verbose: bool = False) -> Path:
    """Compile every CUDA source of the library for sm_100a into one shared object, then the Python entry to it."""
    if force or _lib_stale():
        _build_lib(verbose)
    if force or _ext_stale():
        tmp = str(EXT) + ".tmp"
        subprocess.run(_binding_command(tmp), check=True)
        os.replace(tmp, EXT)
    return LIB


def _build_lib(verbose: bool) -> None:
    objs = []
    build_dir = PKG / "_build"
    build_dir.mkdir(exist_ok=True)
    common = [_nvcc(), "-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a",
              "-Xcompiler", "-fPIC", "-I", str(INCLUDE), "-I", str(CSRC)]
    if verbose:
        common += ["-Xptxas", "-v"]
    procs = []
    for src in SOURCES:
        obj = build_dir / (src + ".o")
        objs.append(str(obj))
        procs.append((src, subprocess.Popen(common + ["-c", str(CSRC / src), "-o", str(obj)],
                                            stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, pr in procs:
        out, _ = pr.communicate()
        if verbose or pr.returncode != 0:
            sys.stderr.write(out)
        failed |= pr.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = str(LIB) + ".tmp"
    subprocess.run([_nvcc(), "-shared", "-Wno-deprecated-gpu-targets", "-o", tmp, *objs, "-cudart", "static"], check=True)
    os.replace(tmp, LIB)


if __name__ == "__main__":
    build(force=True, verbose="-v" in sys.argv)
    print(LIB)
