"""Build libfda.so (sm_100a only) with nvcc and _native.so (its CPython module) next to this file.

Usage: ``python -m paper_2405_20988_b200.build [--force] [--verbose]``
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "libfda.so")
OUT_PY = os.path.join(HERE, "_native.so")
OBJ_DIR = os.path.join(HERE, "_build")
SOURCES = ["fda_api.cu", "fda_hash.cu", "fda_local_state.cu", "fda_local_state_gather.cu", "fda_lanes_12.cu", "fda_lanes_16.cu", "fda_lanes_20.cu", "fda_lanes_22.cu", "fda_lanes_23.cu", "fda_lanes_24.cu", "fda_mean_state_gather.cu", "fda_sched.cu", "fda_local_state_linear.cu", "fda_mean_state.cu", "fda_combine.cu", "fda_average.cu", "fda_noalloc.cu", "fda_probe.cu"]
ARCH = ["-gencode", "arch=compute_100a,code=sm_100a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC"]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _deps_mtime() -> float:
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    files.append(os.path.join(HERE, "..", "include", "fda.h"))
    return max(os.path.getmtime(f) for f in files)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and all(os.path.exists(o) and os.path.getmtime(o) >= _deps_mtime() for o in (OUT, OUT_PY)):
        return OUT
    os.makedirs(OBJ_DIR, exist_ok=True)
    extra = ["-Xptxas", "-v"] if verbose else []

    def compile_one(src: str) -> str:
        obj = os.path.join(OBJ_DIR, src.replace(".cu", ".o"))
        cmd = [_nvcc(), *ARCH, *FLAGS, *extra, "-c", os.path.join(CSRC, src), "-o", obj]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or res.returncode:
            sys.stderr.write(res.stdout + res.stderr)
        if res.returncode:
            raise RuntimeError("nvcc failed on %s" % src)
        return obj

    with ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = OUT + ".tmp%d" % os.getpid()
    subprocess.check_call([_nvcc(), *ARCH, "-shared", "-o", tmp, *objs])
    os.replace(tmp, OUT)
    tmp = OUT_PY + ".tmp%d" % os.getpid()
    subprocess.check_call(["gcc", "-O2", "-Wall", "-shared", "-fPIC", "-I" + sysconfig.get_paths()["include"],
                           os.path.join(CSRC, "fda_py.c"), "-o", tmp, "-L" + HERE, "-l:libfda.so",
                           "-Wl,-rpath,$ORIGIN"])
    os.replace(tmp, OUT_PY)
    return OUT


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
