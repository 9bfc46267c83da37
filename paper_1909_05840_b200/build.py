"""Build libqbert.so in-tree with nvcc for sm_100a, and the Python entry to it, _qbert.so, with the host compiler (no
JIT cache: the built libraries travel with the tree)."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from pathlib import Path

PKG = Path(__file__).resolve().parent
CSRC = PKG / "csrc"
INCLUDE = PKG.parent / "include"
LIB = PKG / "libqbert.so"
EXT = PKG / "_qbert.so"
SOURCES = ["api.cu", "quantize_act.cu", "quantize_weights.cu", "quantize_weights_noalloc.cu", "gemm.cu", "probe.cu", "embedding.cu", "sensitivity.cu"]


def _nvcc() -> str:
    cand = os.environ.get("NVCC") or "/usr/local/cuda/bin/nvcc"
    return cand if Path(cand).exists() else "nvcc"


def needs_build() -> bool:
    if not LIB.exists() or not EXT.exists():
        return True
    t = min(LIB.stat().st_mtime, EXT.stat().st_mtime)
    deps = [d for pattern in ("*.cu", "*.cuh", "*.cpp") for d in CSRC.glob(pattern)] + list(INCLUDE.glob("*.h"))
    return any(d.stat().st_mtime > t for d in deps)


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
    if not force and not needs_build():
        return LIB
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
    tmp = str(EXT) + ".tmp"
    subprocess.run(_binding_command(tmp), check=True)
    os.replace(tmp, EXT)
    return LIB


if __name__ == "__main__":
    build(force=True, verbose="-v" in sys.argv)
    print(LIB)
