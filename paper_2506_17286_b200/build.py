"""Build the CUDA library (sm_100a only) and the extension of its binding next to this file: libgta_b200.so, _gta_binding-*.so.

Usage: python -m paper_2506_17286_b200.build [--force] [--verbose]
nvcc cross-compiles without a GPU; the resulting shared object is loaded by `binding.py`.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
LIB = os.path.join(HERE, "libgta_b200.so")
OBJ_DIR = os.path.join(HERE, "_build")
NATIVE_SRC = os.path.join(CSRC, "gta_binding.cpp")

NVCC_FLAGS = [
    "-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden", "--expt-relaxed-constexpr",
    "-I", INCLUDE, "-I", CSRC,
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def _newest(paths) -> float:
    return max(os.path.getmtime(p) for p in paths)


def native_path() -> str:
    """The binding's extension for this interpreter and its torch, whose C++ interfaces it is built against: another version of
    either looks for a file of its own and never loads this one's."""
    import torch
    return os.path.join(HERE, f"_gta_binding-torch{torch.__version__}-{sys.implementation.cache_tag}.so")


def build_native(force: bool = False) -> str:
    """The binding's extension: plain C++ against the torch of this interpreter."""
    native = native_path()
    sources = [NATIVE_SRC, os.path.join(INCLUDE, "gta.h"), os.path.abspath(__file__)]
    if force or not os.path.exists(native) or os.path.getmtime(native) < _newest(sources):
        import torch
        t = os.path.dirname(torch.__file__)
        cuda = os.path.dirname(os.path.dirname(_nvcc())) or "/usr/local/cuda"
        tmp = native + f".{os.getpid()}.tmp"
        cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
               f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", "-I", INCLUDE]
        for inc in (os.path.join(t, "include"), os.path.join(t, "include", "torch", "csrc", "api", "include"),
                    sysconfig.get_paths()["include"], os.path.join(cuda, "include")):
            cmd += ["-isystem", inc]
        cmd += [NATIVE_SRC, "-o", tmp, "-L", os.path.join(t, "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
        subprocess.check_call(cmd)
        os.replace(tmp, native)
    return native


def build(force: bool = False, verbose: bool = False) -> str:
    sources = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    headers = sorted(glob.glob(os.path.join(CSRC, "*.cuh"))) + [os.path.join(INCLUDE, "gta.h")]
    os.makedirs(OBJ_DIR, exist_ok=True)
    header_time = _newest(headers + [os.path.abspath(__file__)])
    objects, procs = [], []
    for src in sources:
        obj = os.path.join(OBJ_DIR, os.path.basename(src)[:-3] + ".o")
        objects.append(obj)
        if force or not os.path.exists(obj) or os.path.getmtime(obj) < max(os.path.getmtime(src), header_time):
            cmd = [_nvcc(), *NVCC_FLAGS, "-c", src, "-o", obj]
            if verbose:
                cmd.insert(1, "-Xptxas")
                cmd.insert(2, "-v")
            procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if out.strip() and (verbose or p.returncode != 0):
            sys.stderr.write(f"--- {os.path.basename(src)}\n{out}\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    if procs or force or not os.path.exists(LIB) or os.path.getmtime(LIB) < _newest(objects):
        tmp = LIB + f".{os.getpid()}.tmp"
        subprocess.check_call([_nvcc(), "-shared", "-o", tmp, *objects, "-gencode",
                               "arch=compute_100a,code=sm_100a"])
        os.replace(tmp, LIB)
    build_native(force)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
