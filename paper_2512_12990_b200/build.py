"""Builds libslicemoe.so (the C-ABI library, nvcc for sm_100a) and _marshal.so (binding.py's native part) in-tree.

    python -m paper_2512_12990_b200.build [--force] [--verbose]
"""
from __future__ import annotations

import os
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libslicemoe.so")
SOURCES = ["api.cu", "pack.cu", "route.cu", "decode.cu", "batch.cu", "stream.cu", "prefill.cu", "tier.cu", "dbsc.cpp"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC]


# the native argument marshalling of binding.py: a Python extension module against torch's headers
MARSHAL_SRC = os.path.join(CSRC, "marshal.cpp")
MARSHAL = os.path.join(PKG, "_marshal.so")


def _newest_source_mtime() -> float:
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f != "marshal.cpp"] + [os.path.join(ROOT, "include", "slicemoe.h")]
    return max(os.path.getmtime(f) for f in files)


LIB_TRACE = os.path.join(PKG, "libslicemoe_trace.so")


def build(force: bool = False, verbose: bool = False, trace: bool = False) -> str:
    """trace=True builds libslicemoe_trace.so: the same library with the decode kernel's time stamps compiled in
    (-DSLICEMOE_TRACE); the ordinary library is not touched."""
    lib = LIB_TRACE if trace else LIB
    marshal = None if trace else _start_marshal(force)
    if marshal is not None:
        try:
            _build_library(lib, force, verbose, trace)
        finally:
            out, _ = marshal.communicate()
            if marshal.returncode != 0:
                sys.stderr.write(out)
        if marshal.returncode != 0:
            raise RuntimeError("the compiler failed on marshal.cpp")
        os.replace(MARSHAL + ".new", MARSHAL)
        return lib
    return _build_library(lib, force, verbose, trace)


def marshal_tag() -> str:
    """What _marshal.so is compiled against besides its sources: the layouts of torch's and Python's objects."""
    import sysconfig
    import torch
    return f"torch {torch.__version__}, {sysconfig.get_config_var('SOABI')}"


def _marshal_is_current() -> bool:
    deps = (MARSHAL_SRC, os.path.join(ROOT, "include", "slicemoe.h"))
    if not os.path.exists(MARSHAL) or os.path.getmtime(MARSHAL) < max(map(os.path.getmtime, deps)):
        return False
    with open(MARSHAL, "rb") as f:
        return marshal_tag().encode() + b"\0" in f.read()


def _start_marshal(force: bool):
    """Starts the compiler on marshal.cpp when _marshal.so is older than its sources or made for another torch or Python."""
    if not force and _marshal_is_current():
        return None
    import sysconfig
    import torch
    t = os.path.dirname(torch.__file__)
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DSLICEMOE_BUILT_FOR="{marshal_tag()}"', "-I", os.path.join(ROOT, "include"),
           "-isystem", os.path.join(t, "include"), "-isystem", os.path.join(t, "include", "torch", "csrc", "api", "include"),
           "-isystem", cuda, "-isystem", sysconfig.get_paths()["include"], MARSHAL_SRC, "-o", MARSHAL + ".new",
           "-L", os.path.join(t, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python"]
    return subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)


def _build_library(lib: str, force: bool, verbose: bool, trace: bool) -> str:
    if not force and os.path.exists(lib) and os.path.getmtime(lib) >= _newest_source_mtime():
        return lib
    nvcc = os.environ.get("NVCC", "nvcc")
    objs = []
    procs = []
    for src in SOURCES:
        obj = os.path.join(CSRC, os.path.splitext(src)[0] + (".trace.o" if trace else ".o"))
        cmd = [nvcc] + NVCC_FLAGS + (["-DSLICEMOE_TRACE"] if trace else []) + (["-Xptxas", "-v"] if verbose else [])
        cmd += ["-c", os.path.join(CSRC, src), "-o", obj]
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    for src, pr in procs:
        out, _ = pr.communicate()
        if verbose or pr.returncode != 0:
            sys.stderr.write(out)
        if pr.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}")
    cmd = [nvcc, "-shared", "-o", lib] + objs + ["-gencode", "arch=compute_100a,code=sm_100a"]
    subprocess.run(cmd, check=True)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv, trace="--trace" in sys.argv))
