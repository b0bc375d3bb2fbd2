"""Builds the C-ABI shared library (libfly_verify.so) for sm_100a with nvcc,
and the Python extension that marshals its arguments (_native.*.so) with g++.

Both are built in-tree, next to this file.  `python -m
paper_2511_22972_b200.build` rebuilds them; `ensure_built()` rebuilds only what
is older than a source.
"""
from __future__ import annotations

import glob
import importlib.metadata
import os
import shutil
import subprocess
import sys
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG_DIR)
CSRC = os.path.join(PKG_DIR, "csrc")
INCLUDE = os.path.join(ROOT, "include")
LIB_PATH = os.path.join(PKG_DIR, "libfly_verify.so")
NATIVE_SRC = os.path.join(CSRC, "native_binding.cpp")


def _torch_version() -> str:
    try:
        return importlib.metadata.version("torch")
    except importlib.metadata.PackageNotFoundError:  # a source tree on the path
        import torch
        return torch.__version__


# The extension is bound to one Python and one torch: the name says which, so that another one builds its own.
NATIVE_PATH = os.path.join(PKG_DIR, "_native.%s.torch-%s.so" % (sysconfig.get_config_var("SOABI"), _torch_version()))

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-lineinfo", "-std=c++17",
    "-shared", "-Xcompiler", "-fPIC",
    "-cudart", "static",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(INCLUDE, "*.h"))


def _older(path: str, deps) -> bool:
    if not os.path.exists(path):
        return True
    t = os.path.getmtime(path)
    return any(os.path.getmtime(p) > t for p in deps)


def lib_is_stale() -> bool:
    return _older(LIB_PATH, _deps())


def native_is_stale() -> bool:
    return _older(NATIVE_PATH, [NATIVE_SRC] + glob.glob(os.path.join(INCLUDE, "*.h")))


def is_stale() -> bool:
    return lib_is_stale() or native_is_stale()


def nvcc_path() -> str:
    p = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(p):
        raise RuntimeError("nvcc not found: cannot build libfly_verify.so")
    return p


def _run(cmd, path: str, what: str, verbose: bool):
    """Builds `path` beside its place and moves it there, so that processes that build or load it meanwhile see whole files."""
    new = "%s.%d.so" % (path[:-3], os.getpid())
    if verbose:
        print(" ".join([*cmd, "-o", path]), file=sys.stderr)
    try:
        r = subprocess.run([*cmd, "-o", new], capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(what + " failed:\n" + r.stdout + r.stderr)
        os.replace(new, path)
    finally:
        if os.path.exists(new):
            os.remove(new)
    if verbose and (r.stdout or r.stderr):
        print(r.stdout + r.stderr, file=sys.stderr)


def build_lib(verbose: bool = False, extra=()) -> str:
    _run([nvcc_path(), *NVCC_FLAGS, *extra, "-I", INCLUDE, "-I", CSRC, *sources()], LIB_PATH, "nvcc", verbose)
    return LIB_PATH


def build_native(verbose: bool = False) -> str:
    import torch
    root = os.path.dirname(torch.__file__)
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], INCLUDE]
    abi = int(torch._C._GLIBCXX_USE_CXX11_ABI)
    _run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", f"-D_GLIBCXX_USE_CXX11_ABI={abi}",
          *[x for i in inc for x in ("-isystem" if i != INCLUDE else "-I", i)], NATIVE_SRC,
          "-L", os.path.join(root, "lib"), "-lc10", "-ltorch_cpu", "-ltorch_python"], NATIVE_PATH, "g++", verbose)
    return NATIVE_PATH


def build(verbose: bool = False, extra=()) -> str:
    build_native(verbose)
    return build_lib(verbose, extra)


def ensure_built() -> str:
    if native_is_stale():
        build_native()
    if lib_is_stale():
        build_lib()
    return LIB_PATH


if __name__ == "__main__":
    build(verbose=True, extra=["-Xptxas", "-v"] if "-v" in sys.argv else ())
