"""Build the CUDA library (nvcc, sm_100a only, no JIT cache) and the native part of the binding (g++) in-tree."""
from __future__ import annotations

import glob
import os
import subprocess
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libla.so")
FAST_SRC = os.path.join(CSRC, "la_fast.cpp")
FAST = os.path.join(PKG, "_la_fast.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-shared", "--threads", "8",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into paper_2006_16236_b200/libla.so (sm_100a SASS)."""
    if force or _stale():
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        cmd = [nvcc, *NVCC_FLAGS, "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", LIB, *sources()]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        subprocess.run(cmd, check=True)
    build_fast(force)
    return LIB


def _built_for() -> str:
    """What the native part of the binding was compiled against, a string that it carries."""
    import torch
    return f"built for torch {torch.__version__}, {sysconfig.get_config_var('SOABI')}"


def _fast_stale() -> bool:
    """Missing, older than its sources, or compiled against another torch or Python."""
    if not os.path.exists(FAST) or os.path.getmtime(FAST) < max(map(os.path.getmtime, (FAST_SRC, os.path.join(ROOT, "include", "la.h")))):
        return True
    with open(FAST, "rb") as f:
        return _built_for().encode() + b"\0" not in f.read()


def build_fast(force: bool = False) -> str:
    """Compile the native part of the binding against torch's headers; it loads libla.so from its own folder."""
    if force or _fast_stale():
        import torch
        t = os.path.dirname(torch.__file__)
        include = [os.path.join(ROOT, "include"), os.path.join(t, "include"), os.path.join(t, "include", "torch", "csrc", "api", "include"),
                   sysconfig.get_paths()["include"], "/usr/local/cuda/include"]
        cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
               f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DLA_BUILT_FOR="{_built_for()}"', *(f"-I{d}" for d in include), "-o", FAST, FAST_SRC,
               "-L", PKG, "-l:libla.so", "-L", os.path.join(t, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python",
               "-Wl,-rpath,$ORIGIN"]
        subprocess.run(cmd, check=True)
    return FAST


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
