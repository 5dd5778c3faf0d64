"""Builds libtfjsb.so (the CUDA library behind the C ABI of include/tfjsb.h) in-tree with nvcc.

    python -m paper_1901_05350_b200.build [--force] [--verbose]

Target: sm_100a only.  The CUDA runtime is linked statically and the driver API is reached
through cudaGetDriverEntryPoint, so the library loads (and its symbols can be listed) on a
machine without a GPU or driver.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD_DIR = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libtfjsb.so")

SOURCES = [
    "api.cu",
    "executor.cu",
    "elementwise.cu",
    "gemm_fp32_simt.cu",
    "gemm_cta.cu",
    "gemm_pair.cu",
    "gemm_tf32_splitk.cu",
    "conv2d_fp32_simt.cu",
    "depthwise.cu",
    "matmul_static_scratch.cu",
    "dwpw_fused_tcgen05.cu",
    "bf16_storage.cu",
    "backprop.cu",
    "depthwise_grad.cu",
    "conv_grad_tcgen05.cu",
    "conv_patch_tcgen05.cu",
    "gemm_strided_tcgen05.cu",
    "chain_cluster.cu",
]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-std=c++17", "-lineinfo",
    "-Xcompiler", "-fPIC",
    "--fmad=true",
    "-I", INCLUDE, "-I", CSRC,
]


def _nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found")
    return exe


def _newest_dependency() -> float:
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(INCLUDE, "tfjsb.h"), __file__]
    return max(os.path.getmtime(p) for p in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _newest_dependency():
        return LIB
    os.makedirs(BUILD_DIR, exist_ok=True)
    nvcc = _nvcc()
    extra = ["-Xptxas", "-v"] if verbose else []

    def compile_one(src: str) -> str:
        obj = os.path.join(BUILD_DIR, src.replace(".cu", ".o"))
        cmd = [nvcc, *NVCC_FLAGS, *extra, "-c", os.path.join(CSRC, src), "-o", obj]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{res.stdout}\n{res.stderr}")
        if verbose:
            sys.stderr.write(res.stderr)
        return obj

    with ThreadPoolExecutor(max_workers=min(8, len(SOURCES))) as pool:
        objs = list(pool.map(compile_one, SOURCES))
    link = [nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-cudart", "static", "-o", LIB, *objs]
    res = subprocess.run(link, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"link failed:\n{res.stdout}\n{res.stderr}")
    return LIB


BINDING_SRC = os.path.join(PKG, "binding", "fast_calls.cpp")


def binding_path() -> str:
    """The C++ half of the Python binding is compiled against one version of torch and one ABI of Python: its name carries both."""
    import sysconfig

    import torch

    version = "".join(c if c.isalnum() else "_" for c in torch.__version__)
    return os.path.join(PKG, f"_fast_calls_torch{version}{sysconfig.get_config_var('EXT_SUFFIX')}")


def build_binding(force: bool = False) -> str:
    import sysconfig

    import torch

    path = binding_path()
    newest = max(os.path.getmtime(p) for p in (BINDING_SRC, os.path.join(INCLUDE, "tfjsb.h"), __file__))
    if not force and os.path.exists(path) and os.path.getmtime(path) >= newest:
        return path
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(_nvcc()))
    scratch = f"{path}.{os.getpid()}"
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", INCLUDE, "-I", sysconfig.get_paths()["include"], "-I", os.path.join(root, "include"),
           "-I", os.path.join(root, "include", "torch", "csrc", "api", "include"), "-I", os.path.join(cuda, "include"),
           BINDING_SRC, "-o", scratch, "-L", os.path.join(root, "lib"),
           "-ltorch_python", "-ltorch", "-ltorch_cuda", "-lc10", "-lc10_cuda", f"-Wl,-rpath,{os.path.join(root, 'lib')}"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"g++ failed on {BINDING_SRC}:\n{res.stdout}\n{res.stderr}")
    os.replace(scratch, path)
    return path


if __name__ == "__main__":
    path = build(force="--force" in sys.argv, verbose="--verbose" in sys.argv)
    print(path)
    print(build_binding(force="--force" in sys.argv))
