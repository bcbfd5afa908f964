"""Builds libjanus.so (the C-ABI library) in-tree with nvcc for sm_100a, and _native.so (the native half of binding.py) with g++."""
from __future__ import annotations

import importlib.metadata
import importlib.util
import os
import shutil
import subprocess
import sys
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "libjanus.so")
NATIVE_PATH = os.path.join(PKG_DIR, "_native.so")
SOURCES = ["janus_api.cu", "indexer_generic.cu", "indexer_tc.cu", "indexer_tc_batch.cu", "topk.cu", "page_demand.cu", "sparse_attn_generic.cu",
           "sparse_attn_heads.cu", "sparse_attn_latent_pair.cu", "indexer_topk.cu", "diagnostics.cu"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _stale() -> bool:
    if not os.path.exists(LIB_PATH) or not os.path.exists(NATIVE_PATH):
        return True
    t = min(os.path.getmtime(LIB_PATH), os.path.getmtime(NATIVE_PATH))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(PKG_DIR, "..", "include", "janus.h")]
    if any(os.path.getmtime(d) > t for d in deps):
        return True
    with open(NATIVE_PATH, "rb") as f:
        return _native_mark().encode() not in f.read()


def _native_mark() -> str:
    """What _native.so is bound to, and carries as a string: torch's C++ interface and the interpreter's."""
    return f"janus native for torch {importlib.metadata.version('torch')}, {sys.implementation.cache_tag};"


def _native_command() -> list:
    """g++ command for the extension module: torch's C++ headers and libraries are the ones the process has loaded already."""
    torch_dir = list(importlib.util.find_spec("torch").submodule_search_locations)[0]
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(_nvcc())))
    inc = [os.path.join(torch_dir, "include"), sysconfig.get_paths()["include"], os.path.join(cuda, "include")]
    return [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", *[f"-I{d}" for d in inc],
            f'-DJANUS_NATIVE_MARK="{_native_mark()}"', os.path.join(CSRC, "py_binding.cpp"), "-o",
            NATIVE_PATH, "-L" + os.path.join(torch_dir, "lib"), "-ltorch_python", "-ltorch_cpu", "-ltorch", "-lc10", "-lc10_cuda", "-ldl"]


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every kernel for sm_100a into one shared library, and the binding's extension module; returns the library's path."""
    if not force and not _stale():
        return LIB_PATH
    build_dir = os.path.join(PKG_DIR, "build")
    os.makedirs(build_dir, exist_ok=True)
    flags = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC",
             "--expt-relaxed-constexpr", "-Xptxas", "-v" if verbose else "-O3"]
    objs = []
    procs = []
    for src in SOURCES:
        obj = os.path.join(build_dir, src.replace(".cu", ".o"))
        objs.append(obj)
        cmd = [_nvcc(), *flags, "-c", os.path.join(CSRC, src), "-o", obj]
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    procs.append(("py_binding.cpp", subprocess.Popen(_native_command(), stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, pr in procs:
        out, _ = pr.communicate()
        if pr.returncode != 0 or verbose:
            sys.stderr.write(f"--- {src}\n{out}\n")
        failed |= pr.returncode != 0
    if failed:
        raise RuntimeError("compilation failed")
    subprocess.check_call([_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", LIB_PATH, *objs, "-lcudart_static", "-ldl", "-lrt", "-lpthread"])
    return LIB_PATH


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
