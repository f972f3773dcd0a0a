"""Build the CUDA library in-tree with nvcc for sm_100a (cross-compiles without a GPU).

The sources are compiled as separate translation units, in parallel, into objects under ``csrc/build``;
only units whose sources (or any header) changed are recompiled, then everything is linked into
``libtahq.so`` beside this file.  ``_call.so``, the CPython face of the codec calls, is built next to it."""
from __future__ import annotations

import concurrent.futures as cf
import glob
import os
import subprocess
import sysconfig

_PKG = os.path.dirname(os.path.abspath(__file__))
_CSRC = os.path.join(_PKG, "csrc")
_OBJ = os.path.join(_CSRC, "build")
LIB = os.path.join(_PKG, "libtahq.so")
CALL = os.path.join(_PKG, "_call.so")
_CALL_SRC = os.path.join(_CSRC, "call.cpp")
_INCLUDE = os.path.join(os.path.dirname(_PKG), "include")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-fmad=false",            # only the fused multiply-adds written in the source are fused
    "-Xcompiler", "-fPIC",
]


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(_CSRC, "*.cu")))


def _headers() -> list[str]:
    return sorted(glob.glob(os.path.join(_CSRC, "*.cuh")) + glob.glob(os.path.join(_INCLUDE, "*.h")))


def _obj(src: str) -> str:
    return os.path.join(_OBJ, os.path.basename(src)[:-3] + ".o")


def _obj_stale(src: str) -> bool:
    o = _obj(src)
    if not os.path.exists(o):
        return True
    t = os.path.getmtime(o)
    return any(os.path.getmtime(d) > t for d in [src, *_headers()])


def _lib_stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(d) > t for d in [*sources(), *_headers()])


def _call_stale() -> bool:
    if not os.path.exists(CALL):
        return True
    t = os.path.getmtime(CALL)
    return any(os.path.getmtime(d) > t for d in [_CALL_SRC, os.path.join(_INCLUDE, "tahq.h")])


def stale() -> bool:
    return _lib_stale() or _call_stale()


def _build_call() -> None:
    """The extension module finds libtahq.so beside itself."""
    tmp = CALL + f".tmp{os.getpid()}"
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"],
                    "-o", tmp, _CALL_SRC, "-L", _PKG, "-ltahq", "-Wl,-rpath,$ORIGIN"], check=True, cwd=_CSRC)
    os.replace(tmp, CALL)


def build(force: bool = False, verbose: bool = False) -> str:
    if not (force or _lib_stale()):
        if _call_stale():
            _build_call()
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    os.makedirs(_OBJ, exist_ok=True)
    todo = [s for s in sources() if force or _obj_stale(s)]

    def compile_one(src: str) -> str:
        tmp = _obj(src) + f".tmp{os.getpid()}"
        cmd = [nvcc, *NVCC_FLAGS, *(["-Xptxas", "-v"] if verbose else []), "-c", "-o", tmp, src]
        r = subprocess.run(cmd, cwd=_CSRC, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {os.path.basename(src)}:\n{r.stdout}\n{r.stderr}")
        os.replace(tmp, _obj(src))
        return r.stderr

    with cf.ThreadPoolExecutor(max_workers=max(1, min(len(todo), os.cpu_count() or 1))) as ex:
        for log in ex.map(compile_one, todo):
            if verbose and log:
                print(log)
    tmp = LIB + f".tmp{os.getpid()}"
    subprocess.run([nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", tmp,
                    *[_obj(s) for s in sources()]], check=True, cwd=_CSRC)
    os.replace(tmp, LIB)
    if force or _call_stale():
        _build_call()
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
