"""Builds liborthrus.so (sm_100a) with nvcc and the native argument marshalling with g++, in-tree.
Usable without a GPU.  The library needs nvcc alone; without a C++ compiler or torch's headers there is no
native marshalling, and binding.py uses ctypes."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig
import warnings

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "liborthrus.so")
NATIVE_SRC = os.path.join(CSRC, "native_binding.cpp")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr"]


def native_path() -> str:
    """The native marshalling for this interpreter and this torch, whose binary interfaces it is compiled against:
    one file for each pair, so that none is loaded into another."""
    import torch
    return os.path.join(HERE, f"_native.{sys.implementation.cache_tag}-torch{torch.__version__}.so")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def stale_native() -> bool:
    if not os.path.exists(native_path()):
        return True
    t = os.path.getmtime(native_path())
    return any(os.path.getmtime(f) > t for f in [NATIVE_SRC] + glob.glob(os.path.join(ROOT, "include", "*.h")))


def start_native():
    """Starts the compilation of the native argument marshalling (it needs torch's and Python's
    headers and links against torch and liborthrus.so); finish_native() links it."""
    import torch
    inc = os.path.join(os.path.dirname(torch.__file__), "include")
    obj = os.path.join(HERE, "_build", "native_binding.o")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-Wall", "-Wextra",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", os.path.join(ROOT, "include"), "-isystem", inc,
           "-isystem", os.path.join(inc, "torch", "csrc", "api", "include"),
           "-isystem", sysconfig.get_paths()["include"],
           "-isystem", os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include"),
           "-c", NATIVE_SRC, "-o", obj]
    return obj, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)


def finish_native(started) -> None:
    import torch
    obj, pr = started
    out = pr.communicate()[0].decode()
    sys.stderr.write(out)
    if pr.returncode != 0:
        raise RuntimeError("compiling native_binding.cpp failed")
    tmp = native_path() + f".tmp{os.getpid()}"
    subprocess.run([os.environ.get("CXX", "g++"), "-shared", "-o", tmp, obj, "-L", HERE, "-l:liborthrus.so",
                    "-Wl,-rpath,$ORIGIN", "-L", os.path.join(os.path.dirname(torch.__file__), "lib"),
                    "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"], check=True)
    os.replace(tmp, native_path())


def stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + \
        glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(f) > t for f in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    objdir = os.path.join(HERE, "_build")
    os.makedirs(objdir, exist_ok=True)
    native = why = None
    try:
        native = start_native() if force or stale_native() else None
    except OSError as e:                        # no compiler
        why = e
    if force or stale():
        build_lib(objdir, verbose)
    try:
        if native:
            finish_native(native)
    except (RuntimeError, OSError, subprocess.CalledProcessError) as e:
        why = e
    if why:
        warnings.warn(f"no native argument marshalling, calls will go through ctypes: {why}", RuntimeWarning)
    return LIB


def build_lib(objdir: str, verbose: bool) -> None:
    nvcc = os.environ.get("NVCC", "nvcc")
    inc = ["-I", os.path.join(ROOT, "include"), "-I", CSRC]
    procs = []
    objs = []
    for src in sources():
        obj = os.path.join(objdir, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        cmd = [nvcc, *NVCC_FLAGS, *os.environ.get("ORTHRUS_NVCC_EXTRA", "").split(), *inc,
               "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)))
    failed = False
    for src, pr in procs:
        out = pr.communicate()[0].decode()
        if pr.returncode != 0 or verbose:
            sys.stderr.write(f"--- {os.path.basename(src)}\n{out}\n")
        failed |= pr.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = LIB + f".tmp{os.getpid()}"
    subprocess.run([nvcc, "-shared", "-o", tmp, *objs, "-gencode",
                    "arch=compute_100a,code=sm_100a"], check=True)
    os.replace(tmp, LIB)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
