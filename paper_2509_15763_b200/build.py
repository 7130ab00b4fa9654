"""Build the C-ABI shared library ``libunigist.so`` (nvcc, sm_100a) and the Python binding's marshalling module
``_marshal.so`` (g++, against torch) in-tree."""
from __future__ import annotations

import os
import subprocess
import sys
from pathlib import Path

PKG = Path(__file__).resolve().parent
ROOT = PKG.parent
CSRC = PKG / "csrc"
LIB = PKG / "libunigist.so"
MARSHAL = PKG / "_marshal.so"

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr", "-I", str(ROOT / "include"), "-I", str(CSRC),
]


def sources():
    return sorted(CSRC.glob("*.cu"))


def _stale(target: Path, deps) -> bool:
    if not target.exists():
        return True
    t = target.stat().st_mtime
    return any(d.stat().st_mtime > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> Path:
    """Build the library, then the marshalling module that links to it."""
    build_library(force, verbose)
    build_marshal(force)
    return LIB


def build_marshal(force: bool = False) -> Path:
    src = CSRC / "marshal.cpp"
    if not force and not _stale(MARSHAL, [src, ROOT / "include" / "unigist.h"]):
        return MARSHAL
    import sysconfig

    import torch

    t = Path(torch.__file__).resolve().parent
    tmp = MARSHAL.with_suffix(f".tmp{os.getpid()}.so")
    subprocess.check_call([
        os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared",
        f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", "-I", str(ROOT / "include"),
        "-I", str(t / "include"), "-I", str(t / "include" / "torch" / "csrc" / "api" / "include"),
        "-I", "/usr/local/cuda/include", "-I", sysconfig.get_paths()["include"], str(src), "-o", str(tmp),
        "-L", str(PKG), "-l:libunigist.so", "-Wl,-rpath,$ORIGIN", "-L", str(t / "lib"), "-ltorch_python", "-ltorch_cpu",
        "-lc10", "-lc10_cuda"])
    os.replace(tmp, MARSHAL)
    return MARSHAL


def build_library(force: bool = False, verbose: bool = False) -> Path:
    """Compile every .cu under csrc/ into one shared library (objects built in parallel)."""
    deps = list(CSRC.glob("*.cu")) + list(CSRC.glob("*.cuh")) + [ROOT / "include" / "unigist.h"]
    if not force and not _stale(LIB, deps):
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    objdir = PKG / "_build"
    objdir.mkdir(exist_ok=True)
    procs = []
    objs = []
    for src in sources():
        obj = objdir / (src.stem + ".o")
        objs.append(str(obj))
        cmd = [nvcc, *NVCC_FLAGS, "-c", str(src), "-o", str(obj)]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, pr in procs:
        out, _ = pr.communicate()
        if pr.returncode != 0 or verbose:
            print(f"--- {src.name}\n{out}", file=sys.stderr)
        failed |= pr.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = LIB.with_suffix(f".tmp{os.getpid()}.so")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", str(tmp), *objs, "-lcudart_static", "-ldl", "-lpthread", "-lrt"])
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose="-v" in sys.argv)
    print(LIB)
