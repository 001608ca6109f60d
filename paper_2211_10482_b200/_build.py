"""Builds libstructtensor.so (sm_100a, nvcc) and the Python binding _binding.so (g++) in-tree.  Run as a module or call
build()."""
from __future__ import annotations

import concurrent.futures
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
OBJDIR = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libstructtensor.so")
BINDING_SRC = os.path.join(CSRC, "binding.cpp")
BINDING = os.path.join(HERE, "_binding.so")
BINDING_KEY = os.path.join(OBJDIR, "binding.key")      # what _binding.so was built for
# debug build with device-side range checks (-DST_BOUNDS_CHECK; relocatable device code for its one device-wide word)
OBJDIR_CHECK = os.path.join(HERE, "_build_check")
LIB_CHECK = os.path.join(HERE, "libstructtensor_check.so")
CHECK_FLAGS = ["-DST_BOUNDS_CHECK", "-rdc=true"]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC,
]


def _sources():
    return sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def _deps_mtime():
    m = 0.0
    for d in (CSRC, INCLUDE):
        for f in os.listdir(d):
            if f.endswith((".cuh", ".h")):
                m = max(m, os.path.getmtime(os.path.join(d, f)))
    return m


def _compile(src: str, verbose: bool, check: bool = False) -> str:
    obj = os.path.join(OBJDIR_CHECK if check else OBJDIR, src[:-3] + ".o")
    spath = os.path.join(CSRC, src)
    if os.path.exists(obj) and os.path.getmtime(obj) >= max(os.path.getmtime(spath), _deps_mtime()):
        return obj
    cmd = ["nvcc", *NVCC_FLAGS, *(CHECK_FLAGS if check else []), "-c", spath, "-o", obj]
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed for %s:\n%s\n%s" % (src, res.stdout, res.stderr))
    if verbose:
        sys.stderr.write(res.stderr)
    return obj


def _binding_key() -> str:
    """The Python and the torch that a binding is compiled against: it holds for no other."""
    import torch
    return "python %s, torch %s" % (sys.version.split()[0], torch.__version__)


def _build_binding(force: bool) -> None:
    deps = (BINDING_SRC, os.path.join(INCLUDE, "structtensor.h"))
    key = _binding_key()
    built_for = open(BINDING_KEY).read() if os.path.exists(BINDING_KEY) else ""
    if not force and built_for == key and os.path.exists(BINDING) and os.path.getmtime(BINDING) >= max(map(os.path.getmtime, deps)):
        return
    import sysconfig

    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")))
    tmp = BINDING + ".%d.tmp" % os.getpid()
    # the torch libraries are in the process before the module is imported, so no search path is recorded for them
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch._C._GLIBCXX_USE_CXX11_ABI,
           "-I", INCLUDE, "-isystem", os.path.join(root, "include"),
           "-isystem", os.path.join(root, "include", "torch", "csrc", "api", "include"),
           "-isystem", os.path.join(cuda, "include"), "-isystem", sysconfig.get_paths()["include"], BINDING_SRC, "-o", tmp,
           "-L", os.path.join(root, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("g++ failed for binding.cpp:\n%s\n%s" % (res.stdout, res.stderr))
    os.replace(tmp, BINDING)
    os.makedirs(OBJDIR, exist_ok=True)
    with open(BINDING_KEY, "w") as f:
        f.write(key)


def build(force: bool = False, verbose: bool = False, check: bool = False) -> str:
    """Compiles every .cu under csrc/ and links the shared library (check=True: the range-checking debug build), and the
    binding, which both builds are called through."""
    objdir, lib = (OBJDIR_CHECK, LIB_CHECK) if check else (OBJDIR, LIB)
    os.makedirs(objdir, exist_ok=True)
    if force:
        for f in os.listdir(objdir):
            if f.endswith(".o"):
                os.remove(os.path.join(objdir, f))
    srcs = _sources()
    with concurrent.futures.ThreadPoolExecutor(max_workers=min(8, len(srcs) + 1)) as ex:
        binding = ex.submit(_build_binding, force)
        objs = list(ex.map(lambda s: _compile(s, verbose, check), srcs))
    binding.result()
    if force or not os.path.exists(lib) or any(os.path.getmtime(o) > os.path.getmtime(lib) for o in objs):
        tmp = lib + ".%d.tmp" % os.getpid()
        cmd = ["nvcc", "-shared", "-gencode", "arch=compute_100a,code=sm_100a", *(["-rdc=true"] if check else []), "-o", tmp, *objs]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError("link failed:\n%s\n%s" % (res.stdout, res.stderr))
        os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, check="--check" in sys.argv))
