"""Builds libpard.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and the binding's
native marshalling module with the host compiler."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libpard.so")
CALL = os.path.join(HERE, "_pardcall.so")
CALL_SOURCE = os.path.join(CSRC, "pard_pycall.c")
SOURCES = ["pard_pipeline.cu", "pard_plan.cu", "pard_local.cu", "pard_policy.cu", "pard_goodput.cu", "pard_host.cu",
           "pard_static.cu", "pard_wait.cu", "pard_priority.cu", "pard_qdelay.cu", "pard_replay.cu",
           "pard_report.cu"]
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC", "-shared", "-cudart", "static"]


def _inputs():
    files = [os.path.join(CSRC, s) for s in SOURCES]
    files.append(os.path.join(CSRC, "pard_internal.h"))
    files.append(os.path.join(CSRC, "pard_plan_internal.cuh"))
    files.append(os.path.join(CSRC, "pard_direct.cuh"))
    files.append(os.path.join(ROOT, "include", "pard.h"))
    return files


def _older(target, files) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(f) > t for f in files)


def _call_inputs():
    return [CALL_SOURCE, os.path.join(ROOT, "include", "pard.h")]


def stale() -> bool:
    return _older(LIB, _inputs()) or _older(CALL, _call_inputs())


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _older(LIB, _inputs()):
        nvcc = os.environ.get("NVCC", "nvcc")
        tmp = LIB + ".tmp%d" % os.getpid()
        cmd = [nvcc] + FLAGS + (["-Xptxas", "-v"] if verbose else []) + \
              ["-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", tmp] + \
              [os.path.join(CSRC, s) for s in SOURCES]
        subprocess.check_call(cmd)
        os.replace(tmp, LIB)
    if force or _older(CALL, _call_inputs()):
        tmp = CALL + ".tmp%d" % os.getpid()
        subprocess.check_call([os.environ.get("CC", "gcc"), "-O2", "-Wall", "-fPIC", "-shared",
                               "-I", sysconfig.get_paths()["include"], "-I", os.path.join(ROOT, "include"),
                               "-o", tmp, CALL_SOURCE, "-ldl"])
        os.replace(tmp, CALL)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
