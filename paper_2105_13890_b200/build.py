"""Builds libeoq.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and the native part of its Python binding."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from importlib.machinery import EXTENSION_SUFFIXES

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libeoq.so")
# Tagged with the interpreter it is built for: CPython's ABI changes between versions, and another interpreter then builds a
# module of its own instead of loading this one.
BIND = os.path.join(HERE, "_eoqbind" + EXTENSION_SUFFIXES[0])
SOURCES = ["eoq_api.cu", "eoq_igemm.cu", "eoq_igemm_patch.cu", "eoq_igemm_rows.cu", "eoq_wgrad_patch.cu", "eoq_wgrad.cu", "eoq_wgrad_rows.cu", "eoq_finish.cu", "eoq_elementwise.cu", "eoq_update.cu", "eoq_static.cu", "eoq_probe.cu", "eoq_aux.cu", "eoq_pool.cu", "eoq_head.cu", "eoq_bn.cu"]
HEADERS = ["eoq_internal.h", "eoq_cells.cuh", "eoq_device.cuh", "eoq_epilogue.cuh", "eoq_next_head.cuh", os.path.join(ROOT, "include", "eoq.h")]


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, s) for s in SOURCES] + [h if os.path.isabs(h) else os.path.join(CSRC, h) for h in HEADERS]
    return any(os.path.getmtime(d) > t for d in deps)


def build_bind(force: bool = False) -> str:
    """The CPython module behind the entry points called per layer and step; it links against libeoq.so beside it."""
    src = os.path.join(CSRC, "eoq_bind.c")
    header = os.path.join(ROOT, "include", "eoq.h")
    if not force and os.path.exists(BIND) and all(os.path.getmtime(f) <= os.path.getmtime(BIND) for f in (src, header)):
        return BIND
    tmp = BIND + ".%d.tmp" % os.getpid()
    subprocess.check_call([os.environ.get("CC", "gcc"), "-std=c11", "-O2", "-Wall", "-shared", "-fPIC", "-fvisibility=hidden",
                           "-I", os.path.join(ROOT, "include"), "-I", sysconfig.get_paths()["include"], src, "-L", HERE, "-leoq",
                           "-Wl,-rpath,$ORIGIN", "-o", tmp])
    os.replace(tmp, BIND)
    return BIND


def build_lib(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        build_bind()
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + ".%d.tmp" % os.getpid()
    cmd = [nvcc, "-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a",
           "--threads", "0", "-shared", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
           "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-cudart", "static"]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, s) for s in SOURCES] + ["-o", tmp]
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    build_bind(force)
    return LIB


if __name__ == "__main__":
    print(build_lib(force="--force" in sys.argv, verbose="-v" in sys.argv))
