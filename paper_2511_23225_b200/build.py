"""Builds the CUDA library in-tree with nvcc for sm_100a, and the native half of the Python binding with the host
compiler (both without a GPU)."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_HERE)
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "libtweo_b200.so")
NATIVE = os.path.join(_HERE, "_native.so")
SOURCES = ["api.cu", "loss.cu", "block.cu", "absmax.cu", "norm.cu", "quantize.cu", "gemm.cu", "w8a8.cu", "fp4.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC,-fvisibility=hidden", "--expt-relaxed-constexpr"]


def _newer(a: str, b: str) -> bool:
    return not os.path.exists(b) or os.path.getmtime(a) > os.path.getmtime(b)


def native_target() -> str:
    """What the extension module is compiled against beside its sources: torch's C++ interface and Python's C interface."""
    import torch
    return f"torch {torch.__version__} cxx11_abi {int(torch._C._GLIBCXX_USE_CXX11_ABI)} python {sysconfig.get_config_var('EXT_SUFFIX')}"


def build_native(force: bool = False, verbose: bool = False) -> str:
    """The extension module of binding.py (csrc/native.cpp), linked against the library beside it."""
    src, header = os.path.join(CSRC, "native.cpp"), os.path.join(_ROOT, "include", "tweo.h")
    target, stamp = native_target(), os.path.join(_HERE, "_build", "native.target")
    built_for = open(stamp).read() if os.path.exists(stamp) else None
    if force or built_for != target or _newer(src, NATIVE) or _newer(header, NATIVE):
        import torch
        base = os.path.dirname(torch.__file__)
        tmp = NATIVE + f".tmp{os.getpid()}"
        cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
               f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DTWEO_BUILT_FOR="{target}"',
               "-I", os.path.join(_ROOT, "include"), "-isystem", os.path.join(base, "include"),
               "-isystem", os.path.join(base, "include", "torch", "csrc", "api", "include"),
               "-isystem", "/usr/local/cuda/include", "-isystem", sysconfig.get_paths()["include"], src, "-o", tmp,
               "-L", os.path.join(base, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python",
               "-L", _HERE, "-l:" + os.path.basename(LIB), "-Wl,-rpath,$ORIGIN"]
        if verbose:
            sys.stderr.write(" ".join(cmd) + "\n")
        subprocess.check_call(cmd)
        os.replace(tmp, NATIVE)
        os.makedirs(os.path.dirname(stamp), exist_ok=True)
        with open(stamp, "w") as f:
            f.write(target)
    return NATIVE


def build(force: bool = False, verbose: bool = False) -> str:
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    inc = ["-I", os.path.join(_ROOT, "include"), "-I", CSRC]
    objdir = os.path.join(_HERE, "_build")
    os.makedirs(objdir, exist_ok=True)
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    headers.append(os.path.join(_ROOT, "include", "tweo.h"))
    objs, procs = [], []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(objdir, src + ".o")
        objs.append(o)
        if force or _newer(s, o) or any(_newer(h, o) for h in headers):
            cmd = [nvcc, *NVCC_FLAGS, *inc, "-c", s, "-o", o]
            if verbose:
                cmd.insert(1, "-Xptxas")
                cmd.insert(2, "-v")
            procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode:
            sys.stderr.write(f"--- {src}\n{out}\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    if procs or not os.path.exists(LIB):
        tmp = LIB + f".tmp{os.getpid()}"
        subprocess.check_call([nvcc, "-shared", "-o", tmp, *objs, "-gencode", "arch=compute_100a,code=sm_100a",
                               "-Xcompiler", "-fPIC"])
        os.replace(tmp, LIB)
    build_native(force, verbose)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
