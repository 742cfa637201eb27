"""Builds libhoccl.so (sm_100a, nvcc) and the Python call entry points _calls (gcc) in-tree from csrc/.  No JIT cache: both sit next to
this file."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libhoccl.so")
# The name carries the interpreter's ABI (".cpython-312-x86_64-linux-gnu.so"): each interpreter that uses the tree has a module of its
# own and looks for that name before a plain "_calls.so".
CALLS, CALLS_SOURCE = os.path.join(HERE, "_calls" + sysconfig.get_config_var("EXT_SUFFIX")), os.path.join(CSRC, "calls.c")
SOURCES = ["api.cu", "exec.cu", "p2p.cu", "kernels.cu", "plan.cpp", "static_scratch.cu", "proxy.cu", "sched.cpp", "probe.cu", "ring.cu", "graph.cu", "host_entry.cu", "ring_host.cu", "options.cpp", "roles.cu"]
HEADERS = ["comm.h", "kernels.cuh", "device_common.cuh", "plan.h", "proxy.h", "sched.h", "options.h", os.path.join("..", "..", "include", "hoccl.h"), os.path.join("..", "..", "include", "hoccl_diag.h")]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC,-Wall,-Wno-unused-function", "-shared", "-cudart", "static", "--threads", "0",
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def _older(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def is_stale() -> bool:
    return _older(LIB, [os.path.join(CSRC, s) for s in SOURCES + HEADERS] + [os.path.abspath(__file__)])


def build_calls(force: bool = False) -> str:
    """The CPython module that marshals the arguments of the inner-loop calls (csrc/calls.c)."""
    if force or _older(CALLS, [CALLS_SOURCE, os.path.abspath(__file__)]):
        tmp = CALLS + ".tmp.%d" % os.getpid()
        cmd = [os.environ.get("CC", "gcc"), "-O2", "-Wall", "-shared", "-fPIC", "-I" + sysconfig.get_paths()["include"], CALLS_SOURCE, "-o", tmp]
        res = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
        if res.returncode != 0:
            sys.stderr.write(res.stdout)
            raise RuntimeError("gcc failed building " + os.path.basename(CALLS))
        os.replace(tmp, CALLS)
    return CALLS


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile whatever is missing or older than its sources.  Returns the path of the library."""
    build_calls(force)
    if not force and not is_stale():
        return LIB
    tmp = LIB + ".tmp.%d" % os.getpid()
    cmd = [_nvcc()] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + [os.path.join(CSRC, s) for s in SOURCES] + ["-o", tmp]
    res = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout)
        raise RuntimeError("nvcc failed building libhoccl.so")
    if verbose:
        sys.stderr.write(res.stdout)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
