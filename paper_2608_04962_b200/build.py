"""Builds ``libspecroll.so`` (the C-ABI library of sm_100a kernels) in-tree with nvcc."""
from __future__ import annotations

import glob
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libspecroll.so")
LIB_CHECK = os.path.join(HERE, "libspecroll_check.so")   # the same library with the kernels' index checks compiled in
NATIVE_SRC = os.path.join(CSRC, "native.cpp")            # argument marshalling of the Python binding
NATIVE = os.path.join(HERE, "_native.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC"]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(lib=LIB) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + \
        glob.glob(os.path.join(HERE, "..", "include", "*.h"))
    return any(os.path.getmtime(p) > t for p in deps)


def build_native(force: bool = False) -> str:
    """Compile the binding's native part (host code only) against the installed torch.  Returns its path."""
    deps = [NATIVE_SRC, os.path.join(HERE, "..", "include", "specroll.h")]
    if not force and os.path.exists(NATIVE) and all(os.path.getmtime(p) <= os.path.getmtime(NATIVE) for p in deps):
        return NATIVE
    import sysconfig
    import torch
    root = os.path.dirname(os.path.abspath(torch.__file__))
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include")]
    tmp = NATIVE + f".tmp{os.getpid()}"
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared",
                           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
                           "-I" + sysconfig.get_paths()["include"], *[a for d in inc for a in ("-isystem", d)],
                           NATIVE_SRC, "-o", tmp, "-L" + os.path.join(root, "lib"),
                           "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"])
    os.replace(tmp, NATIVE)
    return NATIVE


def build(force: bool = False, verbose: bool = False, check: bool = False) -> str:
    """Compile every kernel for sm_100a and link the shared library.  Returns its path.
    check=True builds the debug variant (-DSPECROLL_CHECK: index checks in the kernels) beside it.
    The binding's native part serves both and is built with the normal one."""
    lib = LIB_CHECK if check else LIB
    if not check:
        build_native(force)
    if not force and not _stale(lib):
        return lib
    objs = []
    procs = []
    bdir = "build_check" if check else "build"
    os.makedirs(os.path.join(HERE, bdir), exist_ok=True)
    flags = list(FLAGS) + os.environ.get("SPECROLL_NVCC_FLAGS", "").split() + (["-DSPECROLL_CHECK"] if check else [])
    if verbose:
        flags = flags + ["-Xptxas", "-v"]
    for src in sources():
        obj = os.path.join(HERE, bdir, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        procs.append((src, subprocess.Popen([NVCC, *flags, "-c", src, "-o", obj],
                                            stdout=subprocess.PIPE, stderr=subprocess.STDOUT)))
    failed = False
    for src, p in procs:
        out = p.communicate()[0].decode()
        if p.returncode != 0 or verbose:
            sys.stderr.write(f"--- {os.path.basename(src)}\n{out}\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = lib + f".tmp{os.getpid()}"
    subprocess.check_call([NVCC, "-shared", "-o", tmp, *objs])
    os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv, check="--check" in sys.argv))
