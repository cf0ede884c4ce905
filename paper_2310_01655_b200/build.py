"""Builds libpsk.so (the C-ABI library) in-tree with nvcc for sm_100a, and _psk_native.so (the Python binding's
argument marshalling, host code only) with g++.

    python -m paper_2310_01655_b200.build [--force] [--verbose]
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libpsk.so")
NATIVE = os.path.join(PKG, "_psk_native.so")
NATIVE_TAG = os.path.join(PKG, "build", "_psk_native.tag")      # what it was built for (binding.native_tag)
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(obj, deps):
    if not os.path.exists(obj):
        return True
    t = os.path.getmtime(obj)
    return any(os.path.getmtime(d) > t for d in deps)


def native_stale():
    """Is _psk_native.so missing, older than its sources, or built for another Python or torch?"""
    from . import binding
    src = os.path.join(CSRC, "psk_binding.cpp")
    try:
        with open(NATIVE_TAG) as f:
            tag = f.read()
    except OSError:
        tag = None
    return tag != binding.native_tag() or _stale(NATIVE, [src, os.path.join(ROOT, "include", "psk.h"), __file__])


def build_native(force=False):
    """Compile csrc/psk_binding.cpp against torch's headers; returns the running compiler or None."""
    if not (force or native_stale()):
        return None
    import sysconfig
    import torch
    from . import binding
    troot = os.path.dirname(torch.__file__)
    os.makedirs(os.path.dirname(NATIVE_TAG), exist_ok=True)
    if os.path.exists(NATIVE_TAG):
        os.remove(NATIVE_TAG)                  # (written again when the compiler has succeeded)
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI), '-DPSK_BUILT_FOR="%s"' % binding.native_tag(),
           "-I", os.path.join(ROOT, "include"), "-I", sysconfig.get_paths()["include"], "-I", os.path.join(troot, "include"),
           "-I", os.path.join(troot, "include", "torch", "csrc", "api", "include"),
           "-I", os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include"),
           os.path.join(CSRC, "psk_binding.cpp"), "-o", NATIVE, "-L", os.path.join(troot, "lib"), "-ltorch_python", "-ltorch_cuda", "-ltorch_cpu", "-ltorch",
           "-lc10_cuda", "-lc10"]
    return subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)


def build(force=False, verbose=False):
    """Compile every .cu under csrc/ and link libpsk.so, and the binding's native part; returns libpsk.so's path."""
    native = build_native(force)
    hdrs = glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h")) + [__file__]
    objdir = os.path.join(PKG, "build")
    os.makedirs(objdir, exist_ok=True)
    objs, procs = [], []
    for src in sources():
        obj = os.path.join(objdir, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if force or _stale(obj, [src] + hdrs):
            cmd = [NVCC] + FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", obj]
            procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write("== %s\n%s\n" % (os.path.basename(src), out))
        failed |= p.returncode != 0
    if native is not None:
        out, _ = native.communicate()
        if native.returncode != 0 or verbose:
            sys.stderr.write("== psk_binding.cpp\n%s\n" % out)
        if native.returncode == 0:
            from . import binding
            with open(NATIVE_TAG, "w") as f:
                f.write(binding.native_tag())
        failed |= native.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    if force or procs or _stale(LIB, objs):
        subprocess.check_call([NVCC, "-shared", "-o", LIB] + objs + ["-lcudart"])
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
