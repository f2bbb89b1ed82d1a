"""Build libhsmm.so in-tree: every csrc/*.cu compiled for sm_103a in parallel, then linked, and
beside it the Python binding's call module (csrc/pycall.c) where Python's headers are installed.

Usage: python -m paper_cs_9809105_gb300.build [--force]
"""
from __future__ import annotations

import concurrent.futures as cf
import glob
import hashlib
import os
import shlex
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "_build")
LIB = os.path.join(OUT, "libhsmm.so")
CALL = os.path.join(OUT, "_hsmmcall" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
INCLUDE = os.path.join(ROOT, "include")

NVCC = os.environ.get("NVCC", os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc"))
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-fno-strict-aliasing",
         f"-I{INCLUDE}", "-diag-suppress", "177"]


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _fingerprint() -> str:
    h = hashlib.sha256()
    for p in _sources() + sorted(glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h"))) + \
            [os.path.join(CSRC, "pycall.c"), os.path.join(INCLUDE, "hsmm.h")]:
        h.update(p.encode())
        with open(p, "rb") as f:
            h.update(f.read())
    h.update(" ".join(ARCH + FLAGS).encode())
    h.update((os.uname().machine + CALL).encode())
    return h.hexdigest()


def compile_call(headers: str, out: str) -> None:
    """The Python binding's call module, with the compiler (and options) of $CC."""
    cmd = shlex.split(os.environ.get("CC") or "gcc") + ["-O2", "-shared", "-fPIC", f"-I{headers}", f"-I{INCLUDE}",
                                                        os.path.join(CSRC, "pycall.c"), "-o", out]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"compiling pycall.c failed:\n{r.stderr}")


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(OUT, exist_ok=True)
    fp = _fingerprint()
    stamp = os.path.join(OUT, "fingerprint")
    headers = sysconfig.get_paths()["include"]
    with_call = os.path.exists(os.path.join(headers, "Python.h"))
    if not force and os.path.exists(LIB) and (os.path.exists(CALL) or not with_call) and \
            os.path.exists(stamp) and open(stamp).read() == fp:
        return LIB
    srcs = _sources()
    objs = [os.path.join(OUT, os.path.basename(s) + ".o") for s in srcs]

    def compile_one(src, obj):
        cmd = [NVCC] + ARCH + FLAGS + ["-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {os.path.basename(src)}:\n{r.stderr}")
        if verbose and r.stderr.strip():
            print(r.stderr, file=sys.stderr)
        return obj

    with cf.ThreadPoolExecutor(max_workers=min(len(srcs), os.cpu_count() or 4)) as ex:
        list(ex.map(compile_one, srcs, objs))
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [NVCC] + ARCH + ["-shared", "-Xcompiler", "-fPIC", "-o", tmp] + objs
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stderr}")
    os.replace(tmp, LIB)
    for old in glob.glob(os.path.join(OUT, "_hsmmcall*.so")):     # of another interpreter or an older library
        os.remove(old)
    if with_call:
        tmp = CALL + f".tmp{os.getpid()}"
        compile_call(headers, tmp)
        os.replace(tmp, CALL)
    with open(stamp, "w") as f:
        f.write(fp)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
