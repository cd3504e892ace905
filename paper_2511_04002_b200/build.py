"""Compile the tsq CUDA library (csrc/*.cu) for sm_100a into paper_2511_04002_b200/libtsq.so, and the torch side of the
binding (csrc/tsq_torch.cpp) into _tsq_torch.so beside it."""
from __future__ import annotations

import glob
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libtsq.so")
TORCH_LIB = os.path.join(HERE, "_tsq_torch.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-fmad=false",              # no implicit FMA contraction: every fused operation in the kernels is explicit
    "-ftz=false", "-prec-div=true", "-prec-sqrt=true",
    "--threads", "0",           # the source files in parallel
    "-shared", "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _newest_input() -> float:
    files = sources() + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh"))
    files += glob.glob(os.path.join(ROOT, "include", "*.h")) + [os.path.abspath(__file__)]
    return max(os.path.getmtime(f) for f in files)


def build(force: bool = False, verbose: bool = False) -> str:
    """Build the shared libraries if missing or stale; return the CUDA library's path."""
    if force or not os.path.exists(LIB) or os.path.getmtime(LIB) < _newest_input():
        _build_cuda(verbose)
    torch_src = os.path.join(CSRC, "tsq_torch.cpp")
    newest = max(os.path.getmtime(f) for f in (torch_src, os.path.join(ROOT, "include", "tsq.h"), os.path.abspath(__file__)))
    if force or not os.path.exists(TORCH_LIB) or os.path.getmtime(TORCH_LIB) < newest:
        _build_torch(torch_src)
    return LIB


def _run(cmd, tmp: str, out: str, what: str) -> str:
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("%s failed:\n%s\n%s\n%s" % (what, " ".join(cmd), res.stdout, res.stderr))
    os.replace(tmp, out)
    return res.stderr


def _build_torch(src: str) -> None:
    import sysconfig

    import torch
    inc = os.path.join(os.path.dirname(torch.__file__), "include")
    libs = os.path.join(os.path.dirname(torch.__file__), "lib")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    tmp = TORCH_LIB + ".tmp.%d" % os.getpid()
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-Wall", "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI)]
    cmd += ["-isystem" + d for d in (inc, os.path.join(inc, "torch", "csrc", "api", "include"), os.path.join(cuda, "include"),
                                     sysconfig.get_paths()["include"])]
    cmd += ["-I", os.path.join(ROOT, "include"), src, "-o", tmp, "-L", HERE, "-ltsq", "-L", libs, "-ltorch_python", "-ltorch_cpu",
            "-lc10_cuda", "-lc10", "-Wl,-rpath,$ORIGIN"]
    _run(cmd, tmp, TORCH_LIB, "g++")


def _build_cuda(verbose: bool) -> None:
    nvcc = os.environ.get("NVCC", "nvcc")
    tmp = LIB + ".tmp.%d" % os.getpid()
    cmd = [nvcc, *NVCC_FLAGS, "-I", os.path.join(ROOT, "include"), "-I", CSRC]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [*sources(), "-o", tmp]
    log = _run(cmd, tmp, LIB, "nvcc")
    if verbose:
        sys.stderr.write(log)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
