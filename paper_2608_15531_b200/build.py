"""Build the C-ABI library ``libfq.so`` (nvcc, sm_100a), its CPython entry ``_fqcall.so`` and the generator's
``libfq_synth.so`` in-tree."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libfq.so")
SOURCES = [os.path.join(CSRC, "fq_host.cpp"), os.path.join(CSRC, "fq_kernels.cu")]
HEADERS = [os.path.join(CSRC, "fq_internal.h"), os.path.join(CSRC, "fq_shares.h"), os.path.join(CSRC, "fq_tc_kernel.cuh"), os.path.join(CSRC, "fq_mma_kernel.cuh"),
           os.path.join(CSRC, "fq_direct_kernel.cuh"), os.path.join(ROOT, "include", "fq.h")]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC,-fopenmp,-ffp-contract=off,-fno-fast-math", "-shared",
    "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


PYCALL = os.path.join(HERE, "_fqcall.so")
PYCALL_SOURCE = os.path.join(CSRC, "fq_pycall.cpp")


def stale(lib: str = LIB, sources=tuple(SOURCES + HEADERS)) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    return any(os.path.getmtime(f) > t for f in sources)


def build_lib(force: bool = False, verbose: bool = False) -> str:
    if force or stale():
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", LIB] + SOURCES + ["-lgomp"]
        subprocess.run(cmd, check=True)
    return LIB


def _built_for(lib: str, tag: str) -> bool:
    """Whether `lib` was compiled with this tag (a string constant of its source)."""
    with open(lib, "rb") as f:
        return tag.encode() + b"\0" in f.read()


def build_pycall(force: bool = False) -> str:
    """The CPython entry to the fused calls: links libfq.so (beside it) and the libraries of the torch that will be
    imported with it, whose C++ interface it uses: it is built anew for another torch."""
    import torch
    tag = f"torch {torch.__version__}"
    if force or stale(PYCALL, (PYCALL_SOURCE, HEADERS[-1])) or not _built_for(PYCALL, tag):
        import sysconfig
        t = os.path.join(os.path.dirname(torch.__file__))
        cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
        cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DFQ_TORCH_TAG="{tag}"',
               "-I", os.path.join(ROOT, "include"), "-I", sysconfig.get_paths()["include"], "-isystem", os.path.join(t, "include"),
               "-isystem", os.path.join(t, "include", "torch", "csrc", "api", "include"), "-isystem", os.path.join(cuda, "include"),
               "-o", PYCALL, PYCALL_SOURCE, "-L", HERE, "-l:libfq.so", "-L", os.path.join(t, "lib"), "-lc10", "-lc10_cuda",
               "-ltorch_cpu", "-ltorch_python", "-Wl,-rpath,$ORIGIN", f"-Wl,-rpath,{os.path.join(t, 'lib')}"]
        subprocess.run(cmd, check=True)
    return PYCALL


def build_all(force: bool = False, verbose: bool = False) -> None:
    build_lib(force, verbose)
    build_pycall(force)
    from . import synth
    synth.build(force)


if __name__ == "__main__":
    sys.path.insert(0, ROOT)
    build_all(force="--force" in sys.argv, verbose="-v" in sys.argv)
    print(LIB)
