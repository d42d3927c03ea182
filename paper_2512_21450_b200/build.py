"""Build librlhead.so (the library, for sm_100a) and _host_calls.*.so (host side of the short calls) in-tree:
python -m paper_2512_21450_b200.build"""
import os
import shutil
import subprocess
import sys
import sysconfig

from .binding import HOST_PATH as HOST_OUT

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
HEADER = os.path.join(ROOT, "include", "rlhead.h")
SRC = os.path.join(CSRC, "rlhead.cu")
OUT = os.path.join(HERE, "librlhead.so")
DEPS = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))] + [HEADER]
HOST_SRC = os.path.join(CSRC, "host_calls.cpp")


def nvcc_path():
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def current(out, deps):
    return os.path.exists(out) and all(os.path.getmtime(out) >= os.path.getmtime(p) for p in deps)


def build_host_calls(force=False):
    if not force and current(HOST_OUT, [HOST_SRC, HEADER]):
        return HOST_OUT
    import torch
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    inc = os.path.join(os.path.dirname(torch.__file__), "include")
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", os.path.join(ROOT, "include"), "-isystem", inc, "-isystem", os.path.join(inc, "torch", "csrc", "api", "include"),
           "-isystem", sysconfig.get_paths()["include"], "-o", HOST_OUT, HOST_SRC,
           "-L", lib, "-lc10", "-ltorch_cpu", "-ltorch_python"]
    subprocess.run(cmd, check=True)
    return HOST_OUT


def build(force=False, verbose=False):
    if not force and current(OUT, DEPS):
        build_host_calls(force)
        return OUT
    cmd = [nvcc_path(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(HERE, "csrc"),
           "-o", OUT, SRC]
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    subprocess.run(cmd, check=True)
    build_host_calls(force)   # last: the library does not need it
    return OUT


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
