"""Builds libccld.so (CUDA, sm_100a) and the binding's _binding module in-tree: python -m paper_2605_04478_b200.build"""
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libccld.so")
SOURCES = [os.path.join(CSRC, "ccld_host.cu"), os.path.join(CSRC, "ccld_static.cu")]
DEPS = SOURCES + [os.path.join(CSRC, f) for f in sorted(os.listdir(CSRC)) if f.endswith(".cuh")] + [
    os.path.join(os.path.dirname(HERE), "include", "ccld.h")]

BINDING_SRC = os.path.join(CSRC, "ccld_binding.cpp")
BINDING = os.path.join(HERE, "_binding" + sysconfig.get_config_var("EXT_SUFFIX"))

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "--shared", "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall", "-Xptxas", "-v"]


def build_binding(force: bool = False) -> str:
    """The CPython module of the binding (g++, the headers of this interpreter and of numpy)."""
    newest = max(os.path.getmtime(p) for p in (BINDING_SRC, DEPS[-1]))
    if not force and os.path.exists(BINDING) and os.path.getmtime(BINDING) >= newest:
        return BINDING
    import numpy
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-Wall", "-I" + sysconfig.get_paths()["include"],
           "-I" + numpy.get_include(), "-o", BINDING, BINDING_SRC]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("the compiler failed: " + " ".join(cmd))
    return BINDING


def build(force: bool = False, verbose: bool = False) -> str:
    build_binding(force)
    newest = max(os.path.getmtime(p) for p in DEPS)
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= newest:
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc] + NVCC_FLAGS + os.environ.get("CCLD_NVCC_EXTRA", "").split() + ["-o", LIB] + SOURCES
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed: " + " ".join(cmd))
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
