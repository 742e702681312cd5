"""Compile in-tree: the CUDA library paper_2308_14711_b200/libfff.so (sm_100a only) and the CPython module torch_call that
makes its tensor-level call."""
from __future__ import annotations

import glob
import os
import re
import shutil
import subprocess
import sys
import sysconfig
import warnings

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libfff.so")
CALL_SRC = os.path.join(CSRC, "torch_call.cpp")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

FLAGS = ["-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
         "-Xcompiler", "-fPIC,-Wall", "-shared", "--expt-relaxed-constexpr"]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return sources() + glob.glob(os.path.join(CSRC, "**", "*.cuh"), recursive=True) + \
        glob.glob(os.path.join(os.path.dirname(HERE), "include", "*.h"))


def up_to_date() -> bool:
    return os.path.exists(LIB) and all(os.path.getmtime(LIB) >= os.path.getmtime(p) for p in _deps())


def build(force: bool = False, verbose: bool = False) -> str:
    if force or not up_to_date():
        tmp = LIB + f".{os.getpid()}.tmp"
        cmd = [NVCC] + FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", tmp] + sources()
        subprocess.check_call(cmd)
        os.replace(tmp, LIB)
    try:
        build_call(force)
    except (OSError, subprocess.CalledProcessError, ImportError) as e:
        warnings.warn(f"torch_call not built ({e}): forward_infer will make its call through ctypes")
    return LIB


def call_lib() -> str:
    """File of the CPython module for this interpreter and this torch: its name carries both, so that a build for another one is
    never loaded (the module uses torch's C++ interface, which changes from version to version)."""
    import torch
    tag = re.sub(r"[^A-Za-z0-9_.+-]", "_", f"{sysconfig.get_config_var('SOABI')}-torch{torch.__version__}")
    return os.path.join(HERE, f"torch_call.{tag}.so")


def cuda_home() -> str:
    """The toolkit that NVCC belongs to (NVCC may be a bare name)."""
    return os.path.dirname(os.path.dirname(os.path.realpath(shutil.which(NVCC) or NVCC)))


def build_call(force: bool = False) -> str:
    """The CPython module (needs torch's headers, not a GPU)."""
    out = call_lib()
    if not force and os.path.exists(out) and os.path.getmtime(out) >= os.path.getmtime(CALL_SRC):
        return out
    import torch
    root = os.path.dirname(torch.__file__)
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           os.path.join(cuda_home(), "include"), sysconfig.get_paths()["include"]]
    tmp = out + f".{os.getpid()}.tmp"
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    cmd += [f"-isystem{d}" for d in inc] + ["-o", tmp, CALL_SRC, "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu",
                                           "-lc10_cuda", "-lc10"]
    subprocess.check_call(cmd)
    os.replace(tmp, out)
    return out


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
    print(call_lib())
