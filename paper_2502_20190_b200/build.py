"""Builds the CUDA library (sm_100a) in-tree: ``python -m paper_2502_20190_b200.build``."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libtj.so")
# entry points for the interpreter that runs this (binding.py): one file per Python version
CALLS = os.path.join(HERE, "_tjcall" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
SOURCES = ["tj_api.cu", "tj_actor.cu", "tj_actor_fma.cu", "tj_learner.cu", "tj_td_fma.cu", "tj_publish.cu", "tj_tc.cu", "tj_tc_actor.cu", "tj_sgd.cu", "tj_sgd_small.cu", "tj_calibrate.cu", "tj_consumer.cu", "tj_split_actor.cu", "tj_sgd_tc.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC",
              "--expt-relaxed-constexpr", "-Wno-deprecated-gpu-targets"]


def _deps():
    out = [os.path.join(HERE, "..", "include", "tj.h")]
    for f in os.listdir(CSRC):
        out.append(os.path.join(CSRC, f))
    return out


def build_calls(force: bool = False) -> str:
    srcs = [os.path.join(CSRC, "tj_python.cpp"), os.path.join(HERE, "..", "include", "tj.h")]
    if force or not os.path.exists(CALLS) or os.path.getmtime(CALLS) < max(os.path.getmtime(p) for p in srcs):
        tmp = CALLS + ".tmp.%d" % os.getpid()
        subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"], srcs[0], "-o", tmp])
        os.replace(tmp, CALLS)
    return CALLS


def compile_library(out: str, bdir: str, more=()) -> str:
    """All sources with the flags above and `more`, objects in `bdir`, linked to `out`."""
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    os.makedirs(bdir, exist_ok=True)
    objs, procs = [], []
    for src in SOURCES:
        obj = os.path.join(bdir, src.replace(".cu", ".o"))
        objs.append(obj)
        cmd = [nvcc] + NVCC_FLAGS + list(more) + ["-c", os.path.join(CSRC, src), "-o", obj]
        procs.append((cmd, subprocess.Popen(cmd)))
    for cmd, pr in procs:
        if pr.wait() != 0:
            raise RuntimeError("nvcc failed: " + " ".join(cmd))
    tmp = out + ".tmp.%d" % os.getpid()
    subprocess.check_call([nvcc, "-shared", "-Wno-deprecated-gpu-targets", "-o", tmp] + objs)
    os.replace(tmp, out)
    return out


def build(force: bool = False, verbose: bool = False) -> str:
    build_calls(force)
    newest = max(os.path.getmtime(p) for p in _deps() if not p.endswith(".cpp"))
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= newest:
        return LIB
    return compile_library(LIB, os.path.join(HERE, "_build"), ["-Xptxas", "-v"] if verbose else [])


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
