"""Build libebd.so (the C ABI of include/ebd.h) for GB300, in-tree.

Each CUDA translation unit is compiled for sm_103a in parallel, then linked
into ``paper_2607_21475_gb300/_build/libebd.so``, which needs the CUDA toolkit
alone.  Where a torch with CUDA is installed, the Python binding's native
marshalling (``csrc/binding.cpp``, against that torch's headers) becomes
``_build/ebd_call.so`` beside it.  Content hashes of the sources and flags (for
the latter also the versions of torch and Python) skip what has not changed.
"""
from __future__ import annotations

import hashlib
import os
import shutil
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(BUILD, "libebd.so")
CALL = os.path.join(BUILD, "ebd_call.so")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "--use_fast_math",
              "-Xptxas", "-O3", "--expt-relaxed-constexpr"]


def _nvcc() -> str:
    cand = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(cand):
        raise RuntimeError("nvcc not found; the CUDA 13 toolkit is required to build libebd")
    return cand


def _sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _torch():
    """The installed torch, None without one or without CUDA in it."""
    try:
        import torch
    except ImportError:
        return None
    return torch if torch.version.cuda else None


def _digest(files, extra) -> str:
    h = hashlib.sha256()
    for f in [*files, os.path.join(INCLUDE, "ebd.h")]:
        h.update(f.encode())
        with open(f, "rb") as fh:
            h.update(fh.read())
    h.update(" ".join(extra).encode())
    return h.hexdigest()


def _lib_digest(extra_flags) -> str:
    return _digest(_sources() + sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC)
                                       if f.endswith((".cuh", ".h"))),
                   ARCH + NVCC_FLAGS + list(extra_flags))


def _call_digest(torch_version: str) -> str:
    return _digest([os.path.join(CSRC, "binding.cpp")],
                   [torch_version, sys.version, sysconfig.get_platform()])


def _fresh(path: str, digest: str) -> bool:
    """Whether `path` was built from what `digest` stands for."""
    stamp = path[:-3] + ".stamp"
    if not (os.path.exists(path) and os.path.exists(stamp)):
        return False
    with open(stamp) as fh:
        return fh.read().strip() == digest


def _stamp(path: str, digest: str) -> None:
    with open(path[:-3] + ".stamp", "w") as fh:
        fh.write(digest)


def _build_call(torch, force: bool) -> None:
    """The native marshalling of ebd.py, against this machine's torch and Python."""
    dig = _call_digest(torch.__version__)
    if not force and _fresh(CALL, dig):
        return
    cuda = os.path.dirname(os.path.dirname(_nvcc()))
    tdir = os.path.dirname(torch.__file__)
    tinc, tlib = os.path.join(tdir, "include"), os.path.join(tdir, "lib")
    inc = [tinc, os.path.join(tinc, "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], os.path.join(cuda, "include")]
    tmp = CALL + ".tmp"
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           *(f"-I{p}" for p in inc), os.path.join(CSRC, "binding.cpp"), "-o", tmp,
           f"-L{tlib}", "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed for binding.cpp:\n{r.stderr}")
    os.replace(tmp, CALL)
    _stamp(CALL, dig)


def build(force: bool = False, verbose: bool = False, extra_flags=()) -> str:
    """Compile the CUDA sources and link libebd.so (and, with a torch to build it
    against, the binding); returns the library path."""
    os.makedirs(BUILD, exist_ok=True)
    torch = _torch()
    dig = _lib_digest(extra_flags)
    if not force and _fresh(LIB, dig):
        if torch is not None:
            _build_call(torch, force)
        return LIB
    nvcc = _nvcc()
    srcs = _sources()
    objs = [os.path.join(BUILD, os.path.basename(s)[:-3] + ".o") for s in srcs]

    def compile_one(src_obj):
        src, obj = src_obj
        cmd = [nvcc, *ARCH, *NVCC_FLAGS, *extra_flags, "-I", INCLUDE, "-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {os.path.basename(src)}:\n{r.stderr}")
        if verbose and r.stderr:
            sys.stderr.write(r.stderr)
        return obj

    with ThreadPoolExecutor(max_workers=min(len(srcs) + 1, os.cpu_count() or 4)) as ex:
        call = ex.submit(_build_call, torch, force) if torch is not None else None
        list(ex.map(compile_one, zip(srcs, objs)))
        if call is not None:
            call.result()
    tmp = LIB + ".tmp"
    cmd = [nvcc, *ARCH, "-shared", "-cudart", "static", "-o", tmp, *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link of libebd.so failed:\n{r.stderr}")
    os.replace(tmp, LIB)
    _stamp(LIB, dig)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
