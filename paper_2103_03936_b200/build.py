"""Builds libpf.so (the C-ABI CUDA library, nvcc for sm_100a) and _pf_native.so (its Python marshalling
module, g++ against torch's headers) in-tree."""
from __future__ import annotations

import importlib.util
import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
OBJ = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libpf.so")
NATIVE = os.path.join(PKG, "_pf_native.so")
NATIVE_KEY = os.path.join(OBJ, "_pf_native.key")      # what _pf_native.so was built against
SOURCES = ["pf_api.cu", "pf_simt.cu", "pf_small.cu", "pf_pack.cu", "pf_tc.cu", "pf_tc_conv.cu", "pf_tc_runs.cu", "pf_tc_any.cu", "pf_tc_conv_res.cu", "pf_tc_conv_bwd.cu", "pf_tc_chain.cu", "pf_tc_chain_multi.cu", "pf_tc_chain_act.cu", "pf_tc_chain_conv.cu", "pf_tc_chain_group.cu", "pf_tc_chain_l2.cu", "pf_tc_pair.cu", "pf_tc_f32.cu", "pf_tc_f32_conv.cu", "pf_static.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC"]


def _mtime(path: str) -> float:
    return os.path.getmtime(path) if os.path.exists(path) else 0.0


def _newest(paths) -> float:
    return max(os.path.getmtime(p) for p in paths)


def _headers():
    return [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".h", ".cuh"))] + [os.path.join(ROOT, "include", "pf.h")]


def nvcc() -> str:
    return os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


def objects(force: bool = False, verbose: bool = False) -> list:
    """The library's objects, compiled where a source or header is newer."""
    sources = [os.path.join(CSRC, s) for s in SOURCES]
    os.makedirs(OBJ, exist_ok=True)
    headers = _newest(_headers())

    def compile_one(src: str) -> str:
        obj = os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")
        if force or _mtime(obj) <= max(headers, os.path.getmtime(src)):
            tmp = obj + f".tmp{os.getpid()}.o"
            subprocess.check_call([nvcc()] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) +
                                  ["-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c", "-o", tmp, src])
            os.replace(tmp, obj)
        return obj

    with ThreadPoolExecutor(max_workers=min(len(sources), os.cpu_count() or 1)) as pool:
        return list(pool.map(compile_one, sources))


def _build_lib(force: bool, verbose: bool) -> None:
    if not force and _mtime(LIB) > _newest([os.path.join(CSRC, s) for s in SOURCES] + _headers()):
        return
    tmp = LIB + f".tmp{os.getpid()}"
    subprocess.check_call([nvcc()] + NVCC_FLAGS + ["-shared", "-o", tmp] + objects(force, verbose))
    os.replace(tmp, LIB)


def _torch_abi() -> int:
    import torch
    return int(torch.compiled_with_cxx11_abi())


def _native_key() -> str:
    """The torch, its C++ ABI and the Python that a built module fits."""
    import torch
    return f"torch {torch.__version__}, cxx11 abi {_torch_abi()}, {sys.implementation.cache_tag}"


def _build_native(force: bool) -> None:
    src = os.path.join(CSRC, "pf_python.cpp")
    key = _native_key()
    built_for = open(NATIVE_KEY).read() if os.path.exists(NATIVE_KEY) else ""
    if not force and built_for == key and _mtime(NATIVE) > _newest([src, os.path.join(ROOT, "include", "pf.h")]):
        return
    torch_dir = os.path.dirname(importlib.util.find_spec("torch").origin)
    cuda = os.path.dirname(os.path.dirname(nvcc()))
    tmp = NATIVE + f".tmp{os.getpid()}"
    includes = [os.path.join(torch_dir, "include"), os.path.join(torch_dir, "include", "torch", "csrc", "api", "include"),
                os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
    subprocess.check_call(
        [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={_torch_abi()}", "-o", tmp, src] +
        [a for d in includes for a in ("-isystem", d)] +
        ["-I", os.path.join(ROOT, "include"), "-L", os.path.join(torch_dir, "lib"), "-L", PKG, "-l:libpf.so", "-ltorch_python", "-ltorch_cuda",
         "-ltorch_cpu", "-ltorch", "-lc10_cuda", "-lc10", "-Wl,-rpath,$ORIGIN"])
    os.replace(tmp, NATIVE)
    os.makedirs(OBJ, exist_ok=True)
    with open(NATIVE_KEY, "w") as f:
        f.write(key)


def build(force: bool = False, verbose: bool = False) -> str:
    _build_lib(force, verbose)
    _build_native(force)
    return LIB


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose="-v" in sys.argv)
    print(LIB)
