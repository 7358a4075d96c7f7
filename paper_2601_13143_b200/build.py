"""Builds ``libfastav.so`` in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the small C module through which
Python calls its hot entry points."""
from __future__ import annotations

import glob
import os
import subprocess
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(_HERE), "include")
LIB_PATH = os.path.join(_HERE, "libfastav.so")
BINDING_SOURCE = os.path.join(CSRC, "binding.c")
BINDING_PATH = os.path.join(_HERE, "_binding" + sysconfig.get_config_var("EXT_SUFFIX"))

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-shared"]


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    built = os.path.getmtime(LIB_PATH)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(INCLUDE, "*.h"))
    return any(os.path.getmtime(f) > built for f in deps)


def build_binding(force: bool = False) -> str:
    newest = max(os.path.getmtime(f) for f in (BINDING_SOURCE, os.path.join(INCLUDE, "fastav.h")))
    if force or not os.path.exists(BINDING_PATH) or newest > os.path.getmtime(BINDING_PATH):
        cc = os.environ.get("CC", "gcc")
        subprocess.run([cc, "-O2", "-shared", "-fPIC", "-Wall", f"-I{INCLUDE}", f"-I{sysconfig.get_paths()['include']}", "-o", BINDING_PATH,
                        BINDING_SOURCE], check=True)
    return BINDING_PATH


def build(force: bool = False, verbose: bool = False) -> str:
    build_binding(force)
    if not force and not _stale():
        return LIB_PATH
    nvcc = os.environ.get("NVCC", "nvcc")
    cmd = [nvcc, *NVCC_FLAGS, f"-I{INCLUDE}", "-o", LIB_PATH, *sources()]
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    subprocess.run(cmd, check=True)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force=True, verbose=True))
