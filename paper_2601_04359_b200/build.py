"""Build the CUDA library in-tree with nvcc for sm_100a (no JIT cache, no torch extension)."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
LIB = os.path.join(HERE, "libpackcache.so")
# the Python binding's native side (csrc/pc_python.cpp); the suffix names the interpreter it is built for
PYLIB = os.path.join(HERE, "_packcache_py" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
SOURCES = ["pc_api.cu", "pc_score.cu", "pc_front.cu", "pc_pack.cu", "pc_attend.cu", "pc_attend_simt.cu", "pc_attend_tc.cu",
           "pc_mass.cu", "pc_host_step.cu", "pc_window.cu", "pc_probe.cu", "pc_probe_tc.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
              "-I", INCLUDE, "-I", CSRC]


def _nvcc() -> str:
    for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if c and (os.path.sep not in c or os.path.exists(c)):
            return c
    raise RuntimeError("nvcc not found")


def _stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(PYLIB):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(PYLIB))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(INCLUDE, "packcache.h"), __file__]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    srcs = [os.path.join(CSRC, s) for s in SOURCES]
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [_nvcc()] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-shared", "-o", tmp] + srcs
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    tmp = PYLIB + f".tmp{os.getpid()}"
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", INCLUDE, "-I", sysconfig.get_paths()["include"],
                           "-o", tmp, os.path.join(CSRC, "pc_python.cpp"), "-L", HERE, "-l:" + os.path.basename(LIB), "-Wl,-rpath,$ORIGIN"])
    os.replace(tmp, PYLIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
