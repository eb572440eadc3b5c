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


def _older(built, deps) -> bool:
    if not all(os.path.exists(f) for f in built):
        return True
    t = min(os.path.getmtime(f) for f in built)
    return any(os.path.getmtime(d) > t for d in deps)


def _stale() -> bool:
    deps = sources() + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) + [os.path.join(CSRC, "calls.cpp")] \
        + glob.glob(os.path.join(ROOT, "include", "*.h")) + [os.path.abspath(__file__)]
    return _older([LIB] + ([CALLS] if HAVE_PYTHON_H else []), deps)


def build_network(force: bool = False) -> bool:
    """Builds csrc/network.cpp where torch's headers are and its version of them compiles; whether there is a module then.  The library works
    without it (the binding has the same in Python), so a compiler's error takes the module away and is not raised."""
    where = torch_dir()
    if not HAVE_PYTHON_H or not where:
        print("no headers of Python or torch: a pruning iteration's table is made in Python", file=sys.stderr)
        return False
    source, include = os.path.join(CSRC, "network.cpp"), os.path.join(where, "include")
    api = os.path.join(include, "torch", "csrc", "api", "include")
    deps = [source, os.path.join(ROOT, "include", "crisp.h"), os.path.abspath(__file__), os.path.join(include, "torch", "csrc", "autograd", "python_variable.h")]
    if not force and not _older([NETWORK], deps):            # (another torch brings newer headers)
        return True
    tmp = NETWORK + f".{os.getpid()}.tmp"
    try:
        subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
                               "-I", PYTHON_INCLUDE, "-I", os.path.join(ROOT, "include"), "-isystem", include, "-isystem", api, "-o", tmp,
                               source, "-L", os.path.join(where, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10"])
        os.replace(tmp, NETWORK)
        return True
    except (subprocess.CalledProcessError, OSError) as e:
        print(f"{source} does not compile against {where} ({e}): a pruning iteration's table is made in Python", file=sys.stderr)
        for f in (tmp, NETWORK):
            if os.path.exists(f):
                os.remove(f)
        return False


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _stale():
        _build_library(verbose)
    build_network(force)
    return LIB


def _build_library(verbose: bool) -> None:
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + f".{os.getpid()}.tmp"
    cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + \
        ["-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", tmp] + sources()
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    if not HAVE_PYTHON_H:
        print(f"no Python.h in {PYTHON_INCLUDE}: the hot calls go through ctypes", file=sys.stderr)
        return
    tmp = CALLS + f".{os.getpid()}.tmp"
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
                           "-I", PYTHON_INCLUDE, "-I", os.path.join(ROOT, "include"), "-o", tmp,
                           os.path.join(CSRC, "calls.cpp")])
    os.replace(tmp, CALLS)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
