"""Builds libtlr.so (the C-ABI routing library) in-tree with nvcc for sm_100a, and the extension module _tlr_torch
(Router.route's marshalling; the package works without it).

    python -m paper_2504_07878_b200.build [--force] [--verbose]
"""
from __future__ import annotations

import glob
import hashlib
import os
import shutil
import subprocess
import sys
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG_DIR)
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "libtlr.so")
TORCH_PATH = os.path.join(PKG_DIR, "_tlr_torch" + sysconfig.get_config_var("EXT_SUFFIX"))
TORCH_KEY = os.path.join(PKG_DIR, "_tlr_torch.key")        # what it was built from
TORCH_SOURCE = os.path.join(CSRC, "tlr_torch.cpp")
TORCH_FLAGS = ["-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden"]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return sources() + sorted(glob.glob(os.path.join(CSRC, "*.cuh"))) + [os.path.join(ROOT, "include", "tlr.h")]


def is_stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    built = os.path.getmtime(LIB_PATH)
    return any(os.path.getmtime(p) > built for p in _deps())


def torch_key() -> str:
    """Everything the extension module depends on: its source, the header whose entry point it calls, torch and the interpreter."""
    import torch
    h = hashlib.sha256()
    for path in (TORCH_SOURCE, os.path.join(ROOT, "include", "tlr.h")):
        with open(path, "rb") as f:
            h.update(f.read())
    return " ".join([h.hexdigest(), torch.__version__, sys.version.split()[0]] + TORCH_FLAGS)


def torch_is_stale() -> bool:
    try:
        with open(TORCH_KEY) as f:
            return f.read() != torch_key() or not os.path.exists(TORCH_PATH)
    except (OSError, ImportError):
        return True


def build_torch() -> str:
    """The extension module: host code only, against the headers of the torch that imports it."""
    import torch
    from torch.utils.cpp_extension import include_paths
    for path in (TORCH_KEY, TORCH_PATH):       # whatever goes wrong: an old one is not used
        if os.path.exists(path):
            os.remove(path)
    libs = os.path.join(os.path.dirname(torch.__file__), "lib")
    cmd = ["g++"] + TORCH_FLAGS + ["-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch.compiled_with_cxx11_abi()),
                                   '-DTLR_TORCH_VERSION="%s"' % torch.__version__,
                                   "-I", os.path.join(ROOT, "include"), "-isystem", sysconfig.get_paths()["include"]]
    for path in include_paths():
        cmd += ["-isystem", path]
    cmd += [TORCH_SOURCE, "-o", TORCH_PATH, "-L", libs, "-ltorch_python", "-ltorch_cpu", "-lc10"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("g++ failed:\n" + res.stdout + res.stderr)
    with open(TORCH_KEY, "w") as f:
        f.write(torch_key())
    return TORCH_PATH


def build(force: bool = False, verbose: bool = False) -> str:
    """Builds what is not up to date; the path of libtlr.so.  Without the extension module everything goes through ctypes, so
    that a machine that cannot build it (no g++, no headers of this interpreter) is told and goes on."""
    path = build_library(force, verbose)
    if force or torch_is_stale():
        try:
            build_torch()
        except Exception as e:      # (an OSError where there is no g++, an ImportError where there is no torch, ...)
            sys.stderr.write("_tlr_torch was not built, Router.route goes through ctypes: %s\n" % e)
    return path


def build_library(force: bool = False, verbose: bool = False) -> str:
    if not force and not is_stale():
        return LIB_PATH
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        raise RuntimeError("nvcc not found; cannot build libtlr.so")
    cmd = [nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
           "-Xcompiler", "-fPIC", "-shared",
           "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", LIB_PATH] + sources()
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + res.stdout + res.stderr)
    if verbose:
        sys.stderr.write(res.stdout + res.stderr)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
