"""Builds, in-tree, libsage.so (the C-ABI library) with nvcc for sm_100a and _native (the marshalling of its calls for
Python) with the host compiler."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG_DIR)
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "libsage.so")
NATIVE_PATH = os.path.join(PKG_DIR, "_native" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
SOURCES = ["tree_ops.cu", "logits_stats.cu", "tree_attention.cu", "tree_attention_rows.cu", "tree_attention_alt.cu", "tree_attention_split.cu"]
NATIVE_SOURCE = "binding.cpp"


def _newest_source_mtime() -> float:
    paths = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(ROOT, "include", "sage.h")]
    return max(os.path.getmtime(p) for p in paths)


def needs_build() -> bool:
    newest = _newest_source_mtime()
    return any(not os.path.exists(p) or os.path.getmtime(p) < newest for p in (LIB_PATH, NATIVE_PATH))


def _run(cmd, what: str, verbose: bool) -> None:
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError(f"building {what} failed")
    if verbose:
        print(res.stderr)


def build_native(verbose: bool = False) -> str:
    """The Python extension; links against libsage.so beside it and against the torch that is installed."""
    import torch
    torch_dir = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    includes = [os.path.join(ROOT, "include"), os.path.join(torch_dir, "include"),
                os.path.join(torch_dir, "include", "torch", "csrc", "api", "include"), sysconfig.get_path("include"),
                os.path.join(cuda, "include")]
    torch_lib = os.path.join(torch_dir, "lib")
    cmd = [os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-shared", "-fPIC", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    for d in includes:
        cmd += ["-isystem" if d != includes[0] else "-I", d]
    cmd += [os.path.join(CSRC, NATIVE_SOURCE), "-o", NATIVE_PATH, LIB_PATH, "-L", torch_lib, "-ltorch_python", "-ltorch_cpu",
            "-lc10_cuda", "-lc10", "-Wl,-rpath,$ORIGIN", f"-Wl,-rpath,{torch_lib}"]
    _run(cmd, "_native", verbose)
    return NATIVE_PATH


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every CUDA source into one shared library, then the Python extension; returns the library's path."""
    if not force and not needs_build():
        return LIB_PATH
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    # (the library's name in the extension's list of needed libraries, found beside it through $ORIGIN)
    cmd = [nvcc, "-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a",
           "-Xcompiler", "-fPIC", "-shared", "-Xlinker", "-soname=libsage.so", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
           "-o", LIB_PATH] + [os.path.join(CSRC, s) for s in SOURCES]
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    _run(cmd, "libsage.so", verbose)
    build_native(verbose)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
