"""Builds libflexiq.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and _calls.so (the Python side's native
marshalling, which links against it and torch) with the host compiler."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig

_DIR = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_DIR)
CSRC = os.path.join(_DIR, "csrc")
LIB = os.path.join(_DIR, "libflexiq.so")
CALLS = os.path.join(_DIR, "_calls.so")
CALLS_FOR = os.path.join(_DIR, "_calls.stamp")   # the Python and torch that _calls.so was built for
SOURCES = ["flexiq_layer.cu", "flexiq_prologue.cu", "flexiq_gemm.cu", "flexiq_reorder.cu", "flexiq_calib.cu", "flexiq_serving.cu", "flexiq_evolution.cu"]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "--fmad=false",  # the epilogue spells out its fused multiply-adds; nothing else may contract
    "-Xcompiler", "-fPIC", "-I", os.path.join(_ROOT, "include"), "-I", CSRC,
]


def _nvcc() -> str:
    """Full path of nvcc; NVCC may be a path or a name to look up."""
    name = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    return shutil.which(name) or name


def _calls_for() -> str:
    import torch
    return f"python {sys.version_info[0]}.{sys.version_info[1]}, torch {torch.__version__}"


def _calls_stale() -> bool:
    if not (os.path.exists(CALLS) and os.path.exists(CALLS_FOR)):
        return True
    with open(CALLS_FOR) as f:
        return f.read() != _calls_for()


def _stale() -> bool:
    if not os.path.exists(LIB) or _calls_stale():
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(CALLS))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(_ROOT, "include", "flexiq.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def build_library(force: bool = False, verbose: bool = False) -> str:
    if not (force or _stale()):
        return LIB
    nvcc = _nvcc()
    objs = []
    for src in SOURCES:
        obj = os.path.join(CSRC, src.replace(".cu", ".o"))
        cmd = [nvcc, *NVCC_FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        subprocess.run(cmd, check=True)
        objs.append(obj)
    subprocess.run([nvcc, "-shared", "-Wno-deprecated-gpu-targets", "-o", LIB, *objs, "-cudart", "static"], check=True)
    _build_calls()
    return LIB


def _build_calls():
    from torch.utils.cpp_extension import include_paths, library_paths
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(_nvcc())))
    include = [sysconfig.get_paths()["include"], *include_paths(), os.path.join(cuda, "include"), os.path.join(_ROOT, "include")]
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", *(f"-I{d}" for d in include), os.path.join(CSRC, "torch_calls.cpp"), "-o", CALLS,
                    f"-L{_DIR}", "-l:libflexiq.so", "-Wl,-rpath,$ORIGIN", *(f"-L{d}" for d in library_paths()), f"-L{os.path.join(cuda, 'lib64')}",
                    "-ltorch_python", "-ltorch", "-ltorch_cpu", "-ltorch_cuda", "-lc10", "-lc10_cuda", "-lcudart"], check=True)
    with open(CALLS_FOR, "w") as f:
        f.write(_calls_for())


if __name__ == "__main__":
    import sys
    print(build_library(force=True, verbose="-v" in sys.argv))
