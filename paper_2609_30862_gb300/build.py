"""In-tree build of the CUDA library (libqieo.so) for sm_103a with nvcc.

One -gencode; the translation units compile in parallel and are linked into one shared
object. The library is rebuilt when a source or the public header is newer than it.
"""
from __future__ import annotations

import glob
import os
import shutil
import subprocess

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(BUILD, "libqieo.so")
GENCODE = "arch=compute_103a,code=sm_103a"


def nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the QIEO CUDA library cannot be built")


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def deps() -> list[str]:
    return sources() + sorted(glob.glob(os.path.join(CSRC, "*.cuh"))) + \
        [os.path.join(ROOT, "include", "qieo.h")]


def stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(d) > t for d in deps())


def objects() -> list[str]:
    """The object of every translation unit, in the order of sources()."""
    return [os.path.join(BUILD, os.path.basename(src)[:-3] + ".o") for src in sources()]


def link(out: str, *more: str) -> None:
    """Link the objects, and whatever else is given, into a shared library."""
    subprocess.check_call([nvcc(), "-gencode", GENCODE, "-shared", *objects(), *more, "-o", out])


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every translation unit to an object in parallel, then link the library."""
    if not force and not stale():
        return LIB
    from concurrent.futures import ThreadPoolExecutor
    os.makedirs(BUILD, exist_ok=True)
    tag = "%d" % os.getpid()
    common = [nvcc(), "-gencode", GENCODE, "-O3", "-lineinfo", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"),
              *(["-Xptxas", "-v"] if verbose else [])]

    def compile_one(pair):
        src, obj = pair
        tmp = obj + ".tmp" + tag
        subprocess.check_call(common + ["-c", src, "-o", tmp])
        os.replace(tmp, obj)

    with ThreadPoolExecutor(max_workers=max(1, len(sources()))) as ex:
        list(ex.map(compile_one, zip(sources(), objects())))
    tmp = LIB + ".tmp" + tag
    link(tmp)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force=True, verbose="-v" in sys.argv))
