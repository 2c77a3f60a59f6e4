"""Compile libowlverify.so (sm_100a, nvcc) and the native half of the Python binding (g++, torch's headers) in-tree.
No GPU needed to build."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "libowlverify.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC", "-shared", "-cudart", "static"]

BINDING = os.path.join(_HERE, "_owl_native.so")
BINDING_SOURCE = os.path.join(CSRC, "torch_binding.cpp")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _run(cmd, target: str) -> None:
    """Compiles to a name of this process's own and moves the result into place (several processes may build at once)."""
    tmp = target + f".tmp{os.getpid()}"
    subprocess.check_call(cmd[:1] + ["-o", tmp] + cmd[1:])
    os.replace(tmp, target)


def build(force: bool = False, verbose: bool = False) -> str:
    """Build what is missing or older than its sources; return the C library's path."""
    header = os.path.join(_HERE, "..", "include", "owlverify.h")
    kernels = [f for f in glob.glob(os.path.join(CSRC, "*")) if f != BINDING_SOURCE] + [header]
    if force or _stale(LIB, kernels):
        _run([NVCC] + FLAGS + (["-Xptxas", "-v"] if verbose else []) + sources(), LIB)
    if force or _stale(BINDING, [BINDING_SOURCE, header]):
        from torch.utils import cpp_extension
        include = [f"-I{d}" for d in cpp_extension.include_paths("cuda") + [sysconfig.get_paths()["include"]]]
        where = [f"-L{d}" for d in cpp_extension.library_paths("cuda") + [_HERE]]
        # the C library is found beside the module; torch's own are in the process already
        _run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", BINDING_SOURCE] + include + where +
             ["-l:libowlverify.so", "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-Wl,-rpath,$ORIGIN"], BINDING)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
