"""Builds the CUDA libraries (sm_100a only, nvcc) and the autograd node (g++) in-tree: ``python -m paper_2510_27527_b200.build``."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libnvfp4_b200.so")
SOURCES = ["api.cu", "quantize.cu", "gemm.cu", "hp.cu", "noalloc.cu", "calib.cu", "osci.cu", "w16.cu", "fp6.cu"]
# measurement aids (the tensor-core issue loop): a library of their own, loaded by the benchmark only
MEASURE_LIB = os.path.join(HERE, "libnvfp4_measure.so")
MEASURE_SOURCES = ["probe.cu"]
# the autograd node of NVFP4Linear: a Python module that calls the library (found beside it) between torch's allocator and engine
NODE_LIB = os.path.join(HERE, "_node.so")
NODE_SOURCES = ["torch_node.cpp"]
HEADERS = ["nvfp4_device.cuh", "nvfp4_internal.h", "nvfp4_tc.cuh", os.path.join("..", "..", "include", "nvfp4.h"),
           os.path.join("..", "..", "include", "nvfp4_measure.h")]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-shared", "--threads", "4",
]


def _stale(lib, sources) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    return any(os.path.getmtime(os.path.join(CSRC, f)) > t for f in sources + HEADERS)


def _compile(lib, sources, verbose):
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = lib + f".{os.getpid()}.tmp"
    cmd = [nvcc] + NVCC_FLAGS + os.environ.get("NVFP4_NVCC_EXTRA", "").split() + (["-Xptxas", "-v"] if verbose else []) + [os.path.join(CSRC, f) for f in sources] + ["-o", tmp]
    subprocess.check_call(cmd)
    os.replace(tmp, lib)


def node_tag() -> str:
    """What the autograd node is compiled against, beside its sources: torch's and Python's binary interfaces have no file to compare."""
    import torch

    return f"torch {torch.__version__}, {sysconfig.get_config_var('SOABI')}"


def _node_stale(lib, sources) -> bool:
    if _stale(lib, sources):
        return True
    with open(lib, "rb") as f:
        return node_tag().encode() + b"\0" not in f.read()  # (the module holds it as `built_for`)


def _compile_node(lib, sources):
    import torch

    at, cuda = os.path.dirname(torch.__file__), os.environ.get("CUDA_HOME", "/usr/local/cuda")
    tmp = lib + f".{os.getpid()}.tmp"
    subprocess.check_call(
        [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
         f'-DNODE_TAG="{node_tag()}"']
        + ["-isystem" + d for d in (f"{at}/include", f"{at}/include/torch/csrc/api/include", f"{cuda}/include", sysconfig.get_paths()["include"])]
        # (the C++ library that torch uses, by name: a compiler that has only the archive would put a second one into the node, whose
        # streams, empty of locale facets, end the process when a message with a number in it is put together)
        + [os.path.join(CSRC, f) for f in sources] + ["-o", tmp, "-l:libstdc++.so.6", f"-L{at}/lib", "-ltorch", "-ltorch_cpu", "-ltorch_python", "-lc10", "-lc10_cuda",
                                                      f"-L{cuda}/lib64", "-lcudart", f"-L{HERE}", "-l:" + os.path.basename(LIB), "-Wl,-rpath,$ORIGIN"])
    os.replace(tmp, lib)


def build(force: bool = False, verbose: bool = False) -> str:
    for lib, sources in ((LIB, SOURCES), (MEASURE_LIB, MEASURE_SOURCES)):
        if force or _stale(lib, sources):
            _compile(lib, sources, verbose)
    if force or _node_stale(NODE_LIB, NODE_SOURCES):
        _compile_node(NODE_LIB, NODE_SOURCES)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
