"""Build libplast.so (the C ABI of include/plast.h) for sm_103a in-tree.

    python -m paper_0804_3643_gb300.build [--verbose]

Each .cu file under csrc/ is compiled in parallel with one -gencode
(compute_103a -> sm_103a), relocatable device code (the score tables live in
constant memory shared across files; the files in WHOLE stand alone), then linked into a shared library next
to this file.  Objects go to csrc/_build/ (git-ignored).
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(CSRC, "_build")
LIB = os.path.join(HERE, "libplast.so")
SOURCES = ["prims.cu", "index.cu", "ungapped.cu", "ungapped_mma.cu", "filter.cu", "gapped.cu", "full.cu", "api.cu", "noalloc.cu"]
# compiled as a whole program: it splits its registers with setmaxnreg, which
# relocatable device code ignores
WHOLE = {"ungapped_mma.cu"}
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    for c in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if c and os.path.exists(c):
            return c
    raise RuntimeError("nvcc not found")


def _flags(verbose: bool, src: str):
    rdc = "-rdc=false" if os.path.basename(src) in WHOLE else "-rdc=true"
    f = ARCH + ["-O3", "-lineinfo", "-std=c++17", rdc, "-Xcompiler", "-fPIC,-O2",
                "-I" + os.path.join(HERE, "..", "include")]
    if verbose:
        f += ["-Xptxas", "-v"]
    return f


def _stale(src: str, obj: str) -> bool:
    if not os.path.exists(obj):
        return True
    t = os.path.getmtime(obj)
    deps = [src] + [os.path.join(CSRC, h) for h in os.listdir(CSRC) if h.endswith(".cuh")]
    deps.append(os.path.join(HERE, "..", "include", "plast.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def build(verbose: bool = False, force: bool = False) -> str:
    os.makedirs(OBJ, exist_ok=True)
    cc = nvcc()
    jobs = []
    for s in SOURCES:
        src = os.path.join(CSRC, s)
        obj = os.path.join(OBJ, s.replace(".cu", ".o"))
        if force or _stale(src, obj):
            jobs.append((src, obj))

    def compile_one(job):
        src, obj = job
        cmd = [cc] + _flags(verbose, src) + ["-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        return src, r

    relink = bool(jobs) or not os.path.exists(LIB)
    with cf.ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        for src, r in ex.map(compile_one, jobs):
            if verbose or r.returncode:
                sys.stderr.write(r.stdout + r.stderr)
            if r.returncode:
                raise RuntimeError(f"nvcc failed on {os.path.basename(src)}")
    if relink:
        objs = [os.path.join(OBJ, s.replace(".cu", ".o")) for s in SOURCES]
        tmp = LIB + f".tmp{os.getpid()}"
        cmd = [cc] + ARCH + ["-shared", "-rdc=true", "-Xcompiler", "-fPIC"] + objs + ["-o", tmp]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("link of libplast.so failed")
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    build(verbose="--verbose" in sys.argv, force="--force" in sys.argv)
    print(LIB)
