"""Builds libreflex_b200.so (the C-ABI library, sm_100a only) and the binding's argument marshalling (_marshal, plain C++) in-tree.

    python -m paper_2607_14695_b200.build [--force] [--verbose]

Extra compiler flags (debug builds with in-kernel timelines: -DREFLEX_TRACE, -DREFLEX_QK_TRACE, -DREFLEX_LIN_TRACE, -DREFLEX_CG_TRACE) can be
given in the environment variable REFLEX_NVCC_FLAGS.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libreflex_b200.so")
MARSHAL_SRC = os.path.join(CSRC, "marshal.cpp")
MARSHAL = os.path.join(HERE, "_marshal" + sysconfig.get_config_var("EXT_SUFFIX"))


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(p) > t for p in deps)


def nvcc_path() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def build_marshal(force: bool = False) -> str:
    """The marshalling module takes the library's symbols from the process (binding.load() opens the library first)."""
    deps = (MARSHAL_SRC, os.path.join(ROOT, "include", "reflex.h"))
    if not force and os.path.exists(MARSHAL) and all(os.path.getmtime(p) <= os.path.getmtime(MARSHAL) for p in deps):
        return MARSHAL
    import torch
    torch_dir = os.path.dirname(torch.__file__)
    tmp = MARSHAL + f".tmp{os.getpid()}"
    cuda = os.path.dirname(os.path.dirname(nvcc_path())) or "/usr/local/cuda"
    inc = [sysconfig.get_paths()["include"], os.path.join(torch_dir, "include"), os.path.join(torch_dir, "include", "torch", "csrc", "api", "include"),
           os.path.join(cuda, "include"), os.path.join(ROOT, "include")]
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"] +
                          [f"-I{p}" for p in inc] + ["-o", tmp, MARSHAL_SRC, "-L" + os.path.join(torch_dir, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"])
    os.replace(tmp, MARSHAL)
    return MARSHAL


def build(force: bool = False, verbose: bool = False) -> str:
    build_marshal(force)
    if not force and not _stale():
        return LIB
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc_path(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
           "-Xcompiler", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
           "--threads", "0", "-o", tmp] + os.environ.get("REFLEX_NVCC_FLAGS", "").split() + sources()
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
        print(" ".join(cmd), file=sys.stderr)
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
