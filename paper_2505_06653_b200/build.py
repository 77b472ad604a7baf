"""Compiles the CUDA sources under ``csrc/`` into ``libbof4.so`` next to this file, and the native
half of the Python binding (``csrc/torch_host.cpp``) into ``_bof4_torch.so``.

sm_100a only.  Both shared libraries are built in-tree so that they travel with the source tree;
they are rebuilt when any source or header is newer than them, and the second one also when it was
built for another torch or Python (it uses torch's C++ interface, which is only stable within a release).
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(_HERE), "include")
LIB = os.path.join(_HERE, "libbof4.so")
HOST_LIB = os.path.join(_HERE, "_bof4_torch.so")
HOST_SRC = os.path.join(CSRC, "torch_host.cpp")
OBJ_DIR = os.path.join(_HERE, "_build")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def _sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _deps():
    hdr = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    hdr += [os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE) if f.endswith(".h")]
    return hdr


def _older(path, deps) -> bool:
    return not os.path.exists(path) or any(os.path.getmtime(p) > os.path.getmtime(path) for p in deps)


def _host_deps():
    return [HOST_SRC] + [os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE) if f.endswith(".h")]


def host_tag() -> str:
    """What the native half of the binding is built for; the module holds it as a string."""
    import torch
    return "bof4 host module for torch %s, Python %s;" % (torch.__version__, sysconfig.get_config_var("SOABI"))


def host_matches(path: str) -> bool:
    """Whether the module at `path` was built for the torch and Python that run now (it is not loaded for this)."""
    with open(path, "rb") as f:
        return host_tag().encode() in f.read()


def _host_stale() -> bool:
    return _older(HOST_LIB, _host_deps()) or not host_matches(HOST_LIB)


def needs_build() -> bool:
    return _older(LIB, _sources() + _deps()) or _host_stale()


def _build_host() -> None:
    """The extension module of the binding: links against torch's libraries and the library next to it."""
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(_nvcc())) or "/usr/local/cuda"
    if not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        cuda = "/usr/local/cuda"
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI), '-DBOF4_HOST_TAG="%s"' % host_tag(), *["-I" + p for p in inc], HOST_SRC,
           "-o", HOST_LIB, "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-ltorch_cuda",
           "-lc10", "-lc10_cuda", "-L" + os.path.join(cuda, "lib64"), "-lcudart", "-L" + _HERE, "-l:" + os.path.basename(LIB),
           "-Wl,-rpath,$ORIGIN"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("g++ failed for %s:\n%s\n%s" % (HOST_SRC, r.stdout, r.stderr))


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    if force or _older(LIB, _sources() + _deps()):
        _build_cuda(force, verbose)
    if force or _host_stale():
        _build_host()
    return LIB


def _build_cuda(force: bool, verbose: bool) -> None:
    os.makedirs(OBJ_DIR, exist_ok=True)
    nvcc = _nvcc()
    hdr_time = max(os.path.getmtime(p) for p in _deps())

    def compile_one(src: str) -> str:
        obj = os.path.join(OBJ_DIR, os.path.basename(src)[:-3] + ".o")
        if (not force and os.path.exists(obj)
                and os.path.getmtime(obj) > max(os.path.getmtime(src), hdr_time)):
            return obj
        cmd = [nvcc, *NVCC_FLAGS, "-I", INCLUDE, "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed for %s:\n%s\n%s" % (src, r.stdout, r.stderr))
        if verbose:
            sys.stderr.write(r.stderr)
        return obj

    with ThreadPoolExecutor(max_workers=8) as ex:
        objs = list(ex.map(compile_one, _sources()))
    cmd = [nvcc, "-shared", "-o", LIB, *objs, "-gencode", "arch=compute_100a,code=sm_100a"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n%s\n%s" % (r.stdout, r.stderr))


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
