"""Builds libsbn.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and the CPython extension that calls it."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG_DIR)
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "libsbn.so")
NATIVE_SOURCE = os.path.join(CSRC, "binding_native.cpp")
NATIVE_PATH = os.path.join(PKG_DIR, "_sbn_native.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-shared", "-Xcompiler", "-fPIC", "-Xptxas", "-v",
]


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh", ".h")))


def needs_build() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    t = os.path.getmtime(LIB_PATH)
    deps = sources() + [os.path.join(ROOT, "include", "sbn.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def build_native(force: bool = False) -> str:
    """Compile csrc/binding_native.cpp into paper_2603_05168_b200/_sbn_native.so.  Returns the path."""
    deps = [NATIVE_SOURCE, os.path.join(ROOT, "include", "sbn.h")]
    if not force and os.path.exists(NATIVE_PATH) and all(os.path.getmtime(d) <= os.path.getmtime(NATIVE_PATH) for d in deps):
        return NATIVE_PATH
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"],
           "-I", os.path.join(ROOT, "include"), "-o", NATIVE_PATH + ".tmp", NATIVE_SOURCE]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("g++ failed building _sbn_native.so")
    os.replace(NATIVE_PATH + ".tmp", NATIVE_PATH)
    return NATIVE_PATH


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile csrc/libsbn.cu into paper_2603_05168_b200/libsbn.so, and the extension.  Returns the library's path."""
    build_native(force)
    if not force and not needs_build():
        return LIB_PATH
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, *NVCC_FLAGS, "-I", os.path.join(ROOT, "include"), "-I", CSRC,
           "-o", LIB_PATH + ".tmp", os.path.join(CSRC, "libsbn.cu")]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed building libsbn.so")
    os.replace(LIB_PATH + ".tmp", LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force=True, verbose=True))
