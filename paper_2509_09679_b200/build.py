"""Builds the CUDA library in-tree, paper_2509_09679_b200/libbfq.so (sm_100a only), and the binding's C++ part beside it."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libbfq.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
         "-Xcompiler", "-fPIC"]


FAST = os.path.join(HERE, "fast_calls" + sysconfig.get_config_var("EXT_SUFFIX"))
FAST_TORCH = os.path.join(HERE, "_build", "fast_calls.torch")  # the torch it was built against


def build_fast_calls(force: bool = False) -> str:
    """The extension module of csrc/fast_calls.cpp (the C ABI's header and torch's)."""
    import torch

    src = os.path.join(CSRC, "fast_calls.cpp")
    newest = max(os.path.getmtime(p) for p in (src, os.path.join(os.path.dirname(HERE), "include", "bfq.h")))
    if not force and os.path.exists(FAST) and os.path.getmtime(FAST) >= newest and os.path.exists(FAST_TORCH):
        with open(FAST_TORCH) as f:
            if f.read() == torch.__version__:
                return FAST
    if os.path.exists(FAST):
        os.remove(FAST)  # what is there is out of date, and stays so if the compiler fails
    at = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(NVCC))
    subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
                    f'-DBFQ_TORCH="{torch.__version__}"',
                    f"-I{at}/include", f"-I{at}/include/torch/csrc/api/include", f"-I{sysconfig.get_paths()['include']}", f"-I{cuda}/include",
                    src, "-o", FAST, f"-L{at}/lib", "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10_cuda", "-lc10"], check=True)
    os.makedirs(os.path.dirname(FAST_TORCH), exist_ok=True)
    with open(FAST_TORCH, "w") as f:
        f.write(torch.__version__)
    return FAST


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + [
        os.path.join(os.path.dirname(HERE), "include", "bfq.h")]


def build(force: bool = False, verbose: bool = False) -> str:
    build_library(force, verbose)
    try:
        build_fast_calls(force)
    except (ImportError, OSError, subprocess.CalledProcessError) as e:  # no C++ compiler, or no headers of Python or torch
        print(f"warning: {FAST} was not built, every call goes through the interpreter: {e}", file=sys.stderr)
    return LIB


def build_library(force: bool = False, verbose: bool = False) -> str:
    newest = max(os.path.getmtime(p) for p in _deps())
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= newest:
        return LIB
    objs = []
    procs = []
    os.makedirs(os.path.join(HERE, "_build"), exist_ok=True)
    for src in sources():
        obj = os.path.join(HERE, "_build", os.path.basename(src) + ".o")
        objs.append(obj)
        if not force and os.path.exists(obj) and os.path.getmtime(obj) >= newest:
            continue
        cmd = [NVCC, *FLAGS, "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write(out)
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    subprocess.run([NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", LIB, *objs,
                    "-cudart", "static"], check=True)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
