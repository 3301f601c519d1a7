"""Compile the CUDA sources into paper_2505_19115_b200/libnvfp4.so (sm_100a only), and the binding's extension module."""
import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
OUT = os.path.join(HERE, "libnvfp4.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


def sources():
    return sorted(glob.glob(os.path.join(HERE, "csrc", "*.cu")))


def _deps():
    return (sources() + glob.glob(os.path.join(HERE, "csrc", "*.cuh")) + glob.glob(os.path.join(HERE, "csrc", "*.h"))
            + [os.path.join(ROOT, "include", "nvfp4.h")])


def _compile(out: str, srcs, defines=(), verbose: bool = False) -> str:
    cmd = [NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
           "--fmad=false",  # every fp32 operation of the quantizer is a single rounding
           "-I", os.path.join(ROOT, "include"), "-o", out] + [f"-D{d}" for d in defines] + list(srcs)
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    subprocess.check_call(cmd)
    return out


def _fresh(out: str, deps=None) -> bool:
    return os.path.exists(out) and all(os.path.getmtime(out) >= os.path.getmtime(d) for d in deps or _deps())


CALLS_OUT = os.path.join(HERE, "_calls.so")
CALLS_BUILT_FOR = os.path.join(HERE, "_calls.so.built_for")     # the Python and PyTorch whose objects the module knows
CALLS_SRC = os.path.join(HERE, "csrc", "python_calls.cpp")


def _text(path: str) -> str:
    if not os.path.exists(path):
        return ""
    with open(path) as f:
        return f.read()


def build_calls(force: bool = False) -> str:
    """The extension module through which binding.py calls the library (host code only)."""
    import torch
    built_for = f"{sysconfig.get_config_var('SOABI')} torch {torch.__version__}"
    if not force and _fresh(CALLS_OUT, [CALLS_SRC, os.path.join(ROOT, "include", "nvfp4.h")]) and _text(CALLS_BUILT_FOR) == built_for:
        return CALLS_OUT
    th = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(NVCC))
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", "-I", os.path.join(th, "include"),
                           "-I", os.path.join(th, "include", "torch", "csrc", "api", "include"),
                           "-I", sysconfig.get_paths()["include"], "-I", os.path.join(cuda, "include"), "-I", os.path.join(ROOT, "include"),
                           CALLS_SRC, "-o", CALLS_OUT, "-L", os.path.join(th, "lib"), "-Wl,-rpath," + os.path.join(th, "lib"),
                           "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python", "-ldl"])
    with open(CALLS_BUILT_FOR, "w") as f:
        f.write(built_for)
    return CALLS_OUT


def build(force: bool = False, verbose: bool = False) -> str:
    if force or not _fresh(OUT):       # first: the C library needs no PyTorch, and is there for C callers whatever becomes of the module
        _compile(OUT, sources(), verbose=verbose)
    build_calls(force)
    return OUT


# Debug build of the same sources with the GEMM's per-role cycle account compiled in (microbench.py gemm_account).
ACCOUNT_OUT = os.path.join(HERE, "libnvfp4_account.so")


def build_account(force: bool = False) -> str:
    if not force and _fresh(ACCOUNT_OUT):
        return ACCOUNT_OUT
    return _compile(ACCOUNT_OUT, sources(), defines=("NVFP4_GEMM_ACCOUNT",))


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
