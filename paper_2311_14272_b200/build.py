"""Build libcrisp.so in-tree with nvcc for sm_100a (cross-compiles without a GPU)."""
from __future__ import annotations

import glob
import importlib.util
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libcrisp.so")
CALLS = os.path.join(HERE, "_calls.so")                      # Python entry points of the hot calls (plain C++)
NETWORK = os.path.join(HERE, "_network.so")                  # and of what goes over the tensors of a network (C++ with torch's headers)
PYTHON_INCLUDE = sysconfig.get_paths()["include"]
HAVE_PYTHON_H = os.path.exists(os.path.join(PYTHON_INCLUDE, "Python.h"))       # without it the binding makes those calls through ctypes


def torch_dir():
    """Where torch is installed with its headers, or None (found without importing it)."""
    spec = importlib.util.find_spec("torch")
    d = os.path.dirname(spec.origin) if spec and spec.origin else None
    return d if d and os.path.exists(os.path.join(d, "include", "torch", "csrc", "autograd", "python_variable.h")) else None

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "--threads", "0", "-shared", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    built = [LIB] + ([CALLS] if HAVE_PYTHON_H else []) + ([NETWORK] if HAVE_PYTHON_H and torch_dir() else [])
    if not all(os.path.exists(f) for f in built):
        return True
    t = min(os.path.getmtime(f) for f in built)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.cpp")) \
        + glob.glob(os.path.join(ROOT, "include", "*.h")) + [os.path.abspath(__file__)]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + f".{os.getpid()}.tmp"
    cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + \
        ["-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", tmp] + sources()
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    if not HAVE_PYTHON_H:
        print(f"no Python.h in {PYTHON_INCLUDE}: the hot calls go through ctypes", file=sys.stderr)
        return LIB
    tmp = CALLS + f".{os.getpid()}.tmp"
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
                           "-I", PYTHON_INCLUDE, "-I", os.path.join(ROOT, "include"), "-o", tmp,
                           os.path.join(CSRC, "calls.cpp")])
    os.replace(tmp, CALLS)
    where = torch_dir()
    if not where:
        print("no headers of torch: a pruning iteration's table is made in Python", file=sys.stderr)
        return LIB
    tmp = NETWORK + f".{os.getpid()}.tmp"
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
                           "-I", PYTHON_INCLUDE, "-I", os.path.join(ROOT, "include"), "-isystem", os.path.join(where, "include"),
                           "-isystem", os.path.join(where, "include", "torch", "csrc", "api", "include"), "-o", tmp,
                           os.path.join(CSRC, "network.cpp"), "-L", os.path.join(where, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10"])
    os.replace(tmp, NETWORK)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
