"""Builds libaircache.so (the sm_100a CUDA library behind the C ABI) in-tree with nvcc."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libaircache.so")
BINDING_SOURCE = os.path.join(CSRC, "binding.c")
BINDING = os.path.join(PKG, "_binding" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
SOURCES = ["api.cu", "score.cu", "score_cluster.cu", "score_dense.cu", "budget.cu", "compact.cu", "decode.cu"]
HEADERS = [os.path.join(CSRC, "common.cuh"), os.path.join(CSRC, "ptx.cuh"), os.path.join(CSRC, "score.cuh"), os.path.join(os.path.dirname(PKG), "include", "aircache.h")]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the AirCache CUDA library cannot be built")


def stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, s) for s in SOURCES] + HEADERS
    return any(os.path.getmtime(d) > t for d in deps)


def build_binding(force: bool = False) -> str | None:
    """Compile the native argument marshalling of the per-token calls (csrc/binding.c) next to this file.  Without it (no C
    compiler, no Python.h) those calls go through ctypes: None then, with a word on why."""
    if not force and os.path.exists(BINDING) and os.path.getmtime(BINDING) >= os.path.getmtime(BINDING_SOURCE):
        return BINDING
    tmp = BINDING + f".tmp{os.getpid()}"
    cc = os.environ.get("CC") or shutil.which("gcc") or shutil.which("cc")
    try:
        if not cc:
            raise OSError("no C compiler found")
        subprocess.check_call([cc, "-O2", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"], BINDING_SOURCE, "-o", tmp])
    except (OSError, subprocess.CalledProcessError) as e:
        print(f"the native marshalling is not built ({e}): the per-token calls go through ctypes", file=sys.stderr)
        return None
    os.replace(tmp, BINDING)
    return BINDING


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu for sm_100a into one shared library next to this file, and the native part of the binding."""
    build_binding(force)
    if not force and not stale():
        return LIB
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-cudart", "static", "--threads", "0"]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += os.environ.get("AIRCACHE_NVCC_FLAGS", "").split()
    cmd += [os.path.join(CSRC, s) for s in SOURCES] + ["-o", tmp]
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="-v" in sys.argv))
