"""Build libptd.so in-tree from csrc/*.cu with nvcc for sm_103a (one -gencode, parallel TUs), and
the Python binding's call module _ptdcall.so from csrc/pycall.cpp."""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
OUT = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libptd.so")
CALLS = os.path.join(PKG, "_ptdcall.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC"]


def nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libptd.so")
    return exe


def _sources():
    return sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def _compile(src: str) -> str:
    obj = os.path.join(OUT, src[:-3] + ".o")
    cmd = [nvcc(), *ARCH, *FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
    return obj


def _compile_calls() -> None:
    tmp = CALLS + ".tmp"
    cmd = [shutil.which("g++") or "g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
           "-I", sysconfig.get_paths()["include"], os.path.join(CSRC, "pycall.cpp"), "-o", tmp, "-ldl"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed on pycall.cpp:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, CALLS)


def build(force: bool = False) -> str:
    """Compile every CUDA source and link the shared library (and the call module); returns its path."""
    os.makedirs(OUT, exist_ok=True)
    srcs = _sources()
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [
        os.path.join(os.path.dirname(PKG), "include", "ptd.h")]
    if not force and os.path.exists(LIB) and os.path.exists(CALLS):
        newest = max(os.path.getmtime(d) for d in deps)
        if min(os.path.getmtime(LIB), os.path.getmtime(CALLS)) >= newest:
            return LIB
    with cf.ThreadPoolExecutor(max_workers=min(8, len(srcs))) as ex:
        calls = ex.submit(_compile_calls)
        objs = list(ex.map(_compile, srcs))
        calls.result()
    tmp = LIB + ".tmp"
    cmd = [nvcc(), *ARCH, "-shared", "-cudart", "static", "-o", tmp, *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force=True))
