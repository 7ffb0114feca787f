"""Builds libbitcos.so (CUDA kernels for sm_100a + host packers, nvcc) and the binding's _calls.so (gcc) in-tree."""
from __future__ import annotations

import os
import shutil
import subprocess
import sysconfig
import tempfile
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libbitcos.so")
CALLS = os.path.join(HERE, "_calls.so")                # the Python binding's entry (csrc/calls.c)
CALLS_SOURCE = os.path.join(CSRC, "calls.c")
INST = os.path.join(CSRC, "gemv_inst.cu")
INST_PARTS = 11             # the parts of gemv_inst.cuh, each compiled by a process of its own
SOURCES = [os.path.join(CSRC, "gemv.cu"), os.path.join(CSRC, "probe.cu"), os.path.join(CSRC, "pack_device.cu"),
           os.path.join(CSRC, "pack.cpp")]
HEADERS = [INST, *(os.path.join(CSRC, h) for h in ("gemv.cuh", "gemv_inst.cuh", "decode.cuh")),
           os.path.join(ROOT, "include", "bitcos.h")]


def nvcc_flags():
    # (only what bitcos.h declares is exported: the statics of inline functions would otherwise be one object for every copy
    # of the library in a process, and a second copy would find the first one's kernels set up)
    return ["-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "--compress-mode=size",
            "-I" + os.path.join(ROOT, "include"), "-Xcompiler", "-fPIC,-fopenmp,-O2,-fvisibility=hidden"]


def compile_library(out, extra=()):
    """Compiles every source (the instantiations part by part) in parallel and links `out`."""
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    jobs = [(INST, ("-DBITCOS_PART=%d" % part,)) for part in range(1, INST_PARTS + 1)] + [(s, ()) for s in SOURCES]
    with tempfile.TemporaryDirectory() as tmp, ThreadPoolExecutor(max(1, min(len(jobs), os.cpu_count() or 1))) as pool:
        objects = [os.path.join(tmp, "%d.o" % i) for i in range(len(jobs))]
        commands = [[nvcc, *nvcc_flags(), *defs, *extra, "-c", "-o", obj, src] for (src, defs), obj in zip(jobs, objects)]
        list(pool.map(subprocess.check_call, commands))
        linked = os.path.join(tmp, "lib.so")
        subprocess.check_call([nvcc, *nvcc_flags(), "-shared", "-o", linked, *objects, "-lgomp"])
        shutil.copy(linked, out)
    return out


def stale(lib=LIB, sources=None) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    return any(os.path.getmtime(f) > t for f in (sources or SOURCES + HEADERS))


def build(force: bool = False, verbose: bool = False) -> str:
    if force or stale():
        compile_library(LIB, ("-Xptxas", "-v") if verbose else ())
    if force or stale(CALLS, [CALLS_SOURCE]):
        subprocess.check_call(["gcc", "-O2", "-fPIC", "-shared", "-Wall", "-I" + sysconfig.get_paths()["include"], "-o", CALLS,
                               CALLS_SOURCE])
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
