"""Build libgpusq.so in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the native part of the
torch binding, _gpusq_torch.so, with the host compiler."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libgpusq.so")
BINDING = os.path.join(HERE, "_gpusq_torch.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
    "-shared", "-Xcompiler", "-fPIC", "-I" + os.path.join(ROOT, "include"), "-I" + CSRC,
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))


def built_for() -> str:
    """What the native part of the binding depends on, written into it: another torch or Python needs another build."""
    import torch

    return "torch %s, Python %d.%d" % (torch.__version__, *sys.version_info[:2])


def _binding_is_stale() -> bool:
    deps = [os.path.join(CSRC, "torch_binding.cpp"), os.path.join(ROOT, "include", "gpusq.h")]
    if not os.path.exists(BINDING) or any(os.path.getmtime(f) > os.path.getmtime(BINDING) for f in deps):
        return True
    with open(BINDING, "rb") as f:
        return built_for().encode() not in f.read()


def build_binding(force: bool = False) -> str:
    """Needs libgpusq.so beside it (found there at run time as well)."""
    if not force and not _binding_is_stale():
        return BINDING
    import torch

    t = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    tmp = BINDING + ".%d.tmp" % os.getpid()
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI), '-DGPUSQ_BUILT_FOR="%s"' % built_for(),
           "-I" + os.path.join(ROOT, "include"), "-I" + os.path.join(t, "include"),
           "-I" + os.path.join(t, "include", "torch", "csrc", "api", "include"),
           "-I" + sysconfig.get_paths()["include"], "-I" + os.path.join(cuda, "include"),
           "-o", tmp, os.path.join(CSRC, "torch_binding.cpp"), "-L" + HERE, "-l:libgpusq.so",
           "-L" + os.path.join(t, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python", "-Wl,-rpath,$ORIGIN"]
    subprocess.run(cmd, check=True)
    os.replace(tmp, BINDING)
    return BINDING


def is_stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(f) > t for f in _deps())


def build(force: bool = False, verbose: bool = False) -> str:
    if force or is_stale():
        nvcc = os.environ.get("NVCC", "nvcc")
        tmp = LIB + ".%d.tmp" % os.getpid()
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", tmp] + sources()
        subprocess.run(cmd, check=True)
        os.replace(tmp, LIB)
    build_binding(force)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
