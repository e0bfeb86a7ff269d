"""Builds ``libnuna.so`` in-tree with nvcc for sm_100a (cross-compiles without a GPU) and, with the host compiler,
``_nuna_py``, the native half of the Python binding."""
from __future__ import annotations

import glob
import importlib.util
import os
import re
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libnuna.so")
NATIVE_SRC = os.path.join(CSRC, "python", "nuna_py.cpp")


def _torch_version() -> str:
    """The installed torch's version, without importing it."""
    path = os.path.join(os.path.dirname(importlib.util.find_spec("torch").origin), "version.py")
    with open(path) as f:
        return re.search(r"^__version__ = ['\"](.+)['\"]", f.read(), re.M).group(1)


def native_path() -> str:
    """Where the marshalling module for this Python and this torch is.  It is compiled against the insides of both, so a
    module built for others has another name and is neither taken for up to date nor loaded."""
    return os.path.join(HERE, f"_nuna_py.torch-{_torch_version()}{sysconfig.get_config_var('EXT_SUFFIX')}")


NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC,-Wall",
    "-shared",
    # IEEE arithmetic: no fast-math, no flush-to-zero, no FMA contraction
    "-ftz=false", "-prec-div=true", "-prec-sqrt=true", "-fmad=false",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cpp")))


def _older(target, deps) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in deps)


def _public_headers():
    return glob.glob(os.path.join(HERE, "..", "include", "*.h"))


def is_stale() -> bool:
    return _older(LIB, sources() + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) + _public_headers())


def _compile(cmd, target: str, verbose: bool) -> None:
    tmp = target + f".tmp{os.getpid()}"
    proc = subprocess.run(cmd + ["-o", tmp], capture_output=True, text=True)
    if proc.returncode != 0:
        sys.stderr.write(proc.stdout + proc.stderr)
        raise RuntimeError(f"{cmd[0]} failed building {os.path.basename(target)}")
    if verbose:
        sys.stderr.write(proc.stderr)
    os.replace(tmp, target)


def build_native(force: bool = False, verbose: bool = False) -> str:
    """The marshalling module: reads addresses and the current stream out of torch's own objects."""
    target = native_path()
    if not force and not _older(target, [NATIVE_SRC] + _public_headers()):
        return target
    torch_dir = os.path.dirname(importlib.util.find_spec("torch").origin)
    inc = os.path.join(torch_dir, "include")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-Wall", "-shared", "-I" + sysconfig.get_paths()["include"]]
    for d in (inc, os.path.join(inc, "torch", "csrc", "api", "include"), os.path.join(cuda, "include")):
        cmd += ["-isystem", d]
    cmd += [NATIVE_SRC, "-L" + os.path.join(torch_dir, "lib"), "-ltorch_python", "-ltorch_cpu", "-ltorch", "-lc10", "-lc10_cuda"]
    _compile(cmd, target, verbose)
    return target


def build(force: bool = False, verbose: bool = False) -> str:
    build_native(force, verbose)
    if not force and not is_stale():
        return LIB
    _compile([os.environ.get("NVCC", "nvcc")] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + sources(), LIB, verbose)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
