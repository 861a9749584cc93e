"""Builds ``libmxint.so`` in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the native half of the binding with
the host compiler against it, torch and the interpreter, whose versions its name carries (``calls_path``)."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libmxint.so")
SOURCES = ["mxint.cu"]


def calls_path() -> str:
    """The native half of the binding for THIS interpreter and torch: another pair finds no file of its name and builds its own."""
    import torch
    return os.path.join(HERE, "_calls-torch%s%s" % (torch.__version__, sysconfig.get_config_var("EXT_SUFFIX")))


def _newest_source_mtime() -> float:
    newest = 0.0
    for root in (CSRC, os.path.join(os.path.dirname(HERE), "include")):
        for name in os.listdir(root):
            if name.endswith((".cu", ".cuh", ".h", ".cpp")):
                newest = max(newest, os.path.getmtime(os.path.join(root, name)))
    return newest


def build(force: bool = False, verbose: bool = False) -> str:
    newest = _newest_source_mtime()

    def current(f: str) -> bool:
        return not force and os.path.exists(f) and os.path.getmtime(f) >= newest

    calls = calls_path()
    if not current(LIB):
        _build_library(verbose)
    elif current(calls):
        return LIB
    _build_calls(calls)
    return LIB


def _build_library(verbose: bool) -> None:
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + ".tmp.%d" % os.getpid()
    cmd = [nvcc, "-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a",
           "-shared", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
           "--expt-relaxed-constexpr", "-o", tmp]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, s) for s in SOURCES]
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)


def _build_calls(path: str) -> None:
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    include = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
               sysconfig.get_paths()["include"], os.path.join(cuda, "include")]
    tmp = path + ".tmp.%d" % os.getpid()
    cmd = [os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-shared", "-fPIC", "-fvisibility=hidden",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI)] + ["-I" + d for d in include]
    cmd += ["-o", tmp, os.path.join(CSRC, "calls.cpp"), "-L" + os.path.join(root, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu",
            "-ltorch_python", "-L" + HERE, "-l:libmxint.so", "-Wl,-rpath,$ORIGIN"]
    subprocess.check_call(cmd)
    os.replace(tmp, path)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
