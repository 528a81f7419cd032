"""In-tree build of the CUDA library ``_lib/libgb300mrt.so`` for sm_103a.

Each translation unit of ``csrc/`` is compiled by nvcc in parallel into ``_build/`` and the
objects are linked into one shared library with a plain C ABI (``include/lbm_mrt.h``). Both
output folders sit inside the package and are git-ignored. Usage::

    python -m paper_2512_16230_gb300.build [--force] [--verbose-ptxas]
"""
from __future__ import annotations

import argparse
import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(PKG, "_build")
LIBDIR = os.path.join(PKG, "_lib")
LIBNAME = "libgb300mrt.so"
LIBPATH = os.path.join(LIBDIR, LIBNAME)

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC",
         "-Xcompiler", "-Wall", "-Xcompiler", "-Wno-implicit-fallthrough", "-I", INCLUDE, "-I", CSRC]


# The step kernels: every fused multiply-add is written out, so that the kernels which share the
# collision (one cell a thread, batched, row-staged) round alike. The few products left on their own
# do not show in the error against FP64 (the collision emulated on the host with contraction on and
# off: 2D vortices and 3D Kolmogorov flows on seven lattices, the same in three digits).
STEP_FLAGS = ["-fmad=false"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA 13 toolkit is required to build the library")


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _deps_mtime():
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE)]
    return max(os.path.getmtime(f) for f in files)


def _compile(src, obj, extra):
    step = STEP_FLAGS if os.path.basename(src).startswith("k_") else []
    cmd = [nvcc()] + ARCH + FLAGS + step + extra + ["-c", src, "-o", obj]
    res = subprocess.run(cmd, capture_output=True, text=True)
    return src, res.returncode, res.stdout + res.stderr


def build(force: bool = False, verbose_ptxas: bool = False, jobs: int | None = None) -> str:
    """Compile every CUDA translation unit for sm_103a and link the shared library."""
    os.makedirs(BUILD, exist_ok=True)
    os.makedirs(LIBDIR, exist_ok=True)
    newest = _deps_mtime()
    srcs = sources()
    objs = [os.path.join(BUILD, os.path.basename(s)[:-3] + ".o") for s in srcs]
    if not force and os.path.exists(LIBPATH) and os.path.getmtime(LIBPATH) >= newest:
        return LIBPATH
    extra = ["-Xptxas", "-v"] if verbose_ptxas else []
    todo = [(s, o) for s, o in zip(srcs, objs)
            if force or verbose_ptxas or not os.path.exists(o) or os.path.getmtime(o) < newest]
    jobs = jobs or min(len(todo) or 1, os.cpu_count() or 4)
    failed = []
    with cf.ThreadPoolExecutor(max_workers=jobs) as ex:
        for src, rc, out in ex.map(lambda so: _compile(so[0], so[1], extra), todo):
            if rc != 0:
                failed.append((src, out))
            elif verbose_ptxas and out.strip():
                sys.stderr.write(f"== {os.path.basename(src)}\n{out}")
    if failed:
        msg = "\n".join(f"--- {os.path.basename(s)}\n{o}" for s, o in failed)
        raise RuntimeError(f"nvcc failed:\n{msg}")
    tmp = LIBPATH + ".tmp"
    cmd = [nvcc()] + ARCH + ["-shared", "-o", tmp] + objs + ["-lcudart_static", "-ldl", "-lrt", "-lpthread"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"link failed:\n{res.stdout}{res.stderr}")
    os.replace(tmp, LIBPATH)
    return LIBPATH


def main(argv=None):
    ap = argparse.ArgumentParser(description=__doc__)
    ap.add_argument("--force", action="store_true")
    ap.add_argument("--verbose-ptxas", action="store_true")
    ap.add_argument("--jobs", type=int, default=None)
    a = ap.parse_args(argv)
    print(build(force=a.force, verbose_ptxas=a.verbose_ptxas, jobs=a.jobs))


if __name__ == "__main__":
    main()
