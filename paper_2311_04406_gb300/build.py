"""Build libmpclinear.so in-tree with nvcc for sm_103a (GB300), and _binding.so,
the native argument marshalling of abi.py, with the host compiler (where Python's
headers are installed; abi.py marshals through ctypes without it).

Each .cu file is compiled to an object in parallel, then linked into one
shared library with the CUDA runtime linked statically.  The build is skipped
when the sources, headers and flags are unchanged (content hash).
"""
from __future__ import annotations

import glob
import hashlib
import os
import shutil
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(ROOT, "_build")
LIB = os.path.join(HERE, "libmpclinear.so")
BINDING = os.path.join(HERE, "_binding.so")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
         "--expt-relaxed-constexpr", "-I" + os.path.join(ROOT, "include")]


def _nvcc() -> str:
    p = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(p):
        raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libmpclinear")
    return p


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _digest(extra=()) -> str:
    h = hashlib.sha256()
    files = _sources() + [os.path.join(CSRC, "binding.c")] + sorted(glob.glob(os.path.join(CSRC, "*.cuh"))) + \
        sorted(glob.glob(os.path.join(CSRC, "*.h"))) + [os.path.join(ROOT, "include", "mpclinear.h")]
    for f in files:
        h.update(f.encode())
        with open(f, "rb") as fh:
            h.update(fh.read())
    h.update(" ".join(ARCH + FLAGS + list(extra) + [sys.version]).encode())
    return h.hexdigest()


def binding_headers():
    """The folder of Python.h, or None."""
    inc = sysconfig.get_paths()["include"]
    return inc if os.path.exists(os.path.join(inc, "Python.h")) else None


def build_binding(headers):
    """Compile _binding.so; without Python's headers only an older one is removed."""
    if not headers:
        if os.path.exists(BINDING):
            os.remove(BINDING)
        return
    cc = shutil.which("gcc") or shutil.which("cc")
    if not cc:
        raise RuntimeError("a C compiler is required to build the binding")
    tmp = BINDING + f".{os.getpid()}.tmp"
    r = subprocess.run([cc, "-O2", "-fPIC", "-shared", "-I" + os.path.join(ROOT, "include"), "-I" + headers, "-o", tmp,
                        os.path.join(CSRC, "binding.c"), "-ldl"], capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"the binding does not compile:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, BINDING)


def build(force: bool = False, verbose: bool = False, extra_flags=()) -> str:
    nvcc = _nvcc()
    os.makedirs(BUILD, exist_ok=True)
    stamp = os.path.join(BUILD, "libmpclinear.sha256")
    dig = _digest(extra_flags)
    headers = binding_headers()
    if not force and os.path.exists(LIB) and (os.path.exists(BINDING) or not headers) and \
            os.path.exists(stamp) and open(stamp).read() == dig:
        return LIB

    def compile_one(src):
        obj = os.path.join(BUILD, os.path.basename(src)[:-3] + ".o")
        cmd = [nvcc] + ARCH + FLAGS + list(extra_flags) + ["-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {os.path.basename(src)}:\n{r.stdout}\n{r.stderr}")
        if verbose and (r.stdout or r.stderr):
            print(r.stdout + r.stderr)
        return obj

    srcs = _sources()
    with ThreadPoolExecutor(max_workers=min(8, len(srcs))) as ex:
        objs = list(ex.map(compile_one, srcs))
    tmp = LIB + f".{os.getpid()}.tmp"
    r = subprocess.run([nvcc] + ARCH + ["-shared", "-cudart", "static", "-o", tmp] + objs,
                       capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    build_binding(headers)
    with open(stamp, "w") as fh:
        fh.write(dig)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
