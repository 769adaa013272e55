"""Builds libamskv.so in-tree with nvcc for sm_100a (no JIT cache, no torch extension), and the small CPython module
(_steps) through which the binding calls it."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libamskv.so")
STEPS = os.path.join(HERE, "_steps" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
STEPS_SOURCE = os.path.join(CSRC, "steps.c")
SOURCES = ["api.cu", "append.cu", "attend_simt.cu", "attend_tc.cu", "attend_pair.cu", "attend_small.cu", "attend_mid.cu", "similarity.cu", "density.cu", "selftest.cu"]
HEADERS = ["kernels.cuh", "policy.hpp", "sm100_ptx.cuh", os.path.join("..", "..", "include", "amskv.h")]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden", "--expt-relaxed-constexpr"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, s) for s in SOURCES + HEADERS] + [os.path.abspath(__file__)]
    return any(os.path.getmtime(d) > t for d in deps)


def build_steps(force: bool = False) -> str:
    """Compile the binding's CPython module for the running interpreter."""
    if not force and os.path.exists(STEPS) and os.path.getmtime(STEPS) >= os.path.getmtime(STEPS_SOURCE):
        return STEPS
    tmp = STEPS + ".tmp.%d" % os.getpid()
    try:
        subprocess.check_call([os.environ.get("CC", "gcc"), "-O2", "-shared", "-fPIC", "-fvisibility=hidden",
                               "-I" + sysconfig.get_paths()["include"], STEPS_SOURCE, "-o", tmp])
    except (OSError, subprocess.CalledProcessError) as e:
        # no C compiler or no Python headers here: the binding then goes through ctypes alone
        sys.stderr.write("_steps not built (%s): the calls of a step go through ctypes\n" % e)
        if os.path.exists(STEPS):
            os.remove(STEPS)   # not one of older sources
        return ""
    os.replace(tmp, STEPS)
    return STEPS


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu for sm_100a into one shared library next to this file."""
    build_steps(force)
    if not force and not _stale():
        return LIB
    objs = []
    build_dir = os.path.join(HERE, "_build")
    os.makedirs(build_dir, exist_ok=True)
    procs = []
    for s in SOURCES:
        obj = os.path.join(build_dir, s.replace(".cu", ".o"))
        cmd = [_nvcc()] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", os.path.join(CSRC, s), "-o", obj]
        procs.append((s, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    failed = False
    for s, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write("[%s]\n%s\n" % (s, out))
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = LIB + ".tmp.%d" % os.getpid()
    subprocess.check_call([_nvcc(), "-shared", "-o", tmp] + objs + ["-Xcompiler", "-fvisibility=hidden"])
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="-v" in sys.argv))
