"""Builds the native code in-tree: libsnapkv.so (nvcc, sm_100a) and _native.so, the CPython
extension that the binding calls it through (g++).

    python -m paper_2404_14469_b200.build [--force] [--verbose]
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "build")
LIB = os.path.join(HERE, "libsnapkv.so")
NATIVE = os.path.join(HERE, "_native.so")
SOURCES = ["snapkv_api.cu", "snapkv_score.cu", "snapkv_select.cu", "snapkv_select_cluster.cu", "snapkv_gather.cu",
           "snapkv_metrics.cu", "snapkv_decode.cu", "snapkv_score_ragged.cu"]
HEADERS = ["sm100_ptx.cuh", "score_kernel.cuh", "snapkv_internal.h", "launch.cuh", "snapkv_binding.h", os.path.join("..", "..", "include", "snapkv.h")]
NATIVE_SOURCE = "native_binding.cpp"
NATIVE_HEADERS = ["snapkv_binding.h", os.path.join("..", "..", "include", "snapkv.h")]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: libsnapkv.so cannot be built")


def _older(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(os.path.join(CSRC, d)) > t for d in deps)


def _run(cmd, what: str, verbose: bool):
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"{what} failed:\n" + res.stdout + res.stderr)
    if verbose:
        sys.stderr.write(res.stdout + res.stderr)
    return res.stdout + res.stderr


def _build_lib(force: bool, verbose: bool):
    """One object per source, compiled side by side, then one shared library.  What ptxas says of each
    kernel's registers and spills stays beside the object (build/<source>.ptxas)."""
    if not force and not _older(LIB, SOURCES + HEADERS):
        return
    os.makedirs(OBJ, exist_ok=True)
    flags = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
             "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC,-O3,-Wall", "-Xptxas", "-v"]

    def compile_one(src):
        obj = os.path.join(OBJ, src + ".o")
        if force or _older(obj, [src] + HEADERS):
            said = _run([_nvcc(), "-c", *flags, "-o", obj, os.path.join(CSRC, src)], "nvcc " + src, verbose)
            with open(os.path.join(OBJ, src + ".ptxas"), "w") as f:
                f.write(said)
        return obj

    with ThreadPoolExecutor(max_workers=min(len(SOURCES), os.cpu_count() or 1)) as pool:
        objs = list(pool.map(compile_one, SOURCES))
    _run([_nvcc(), "-shared", "-o", LIB, "-gencode", "arch=compute_100a,code=sm_100a", "-cudart", "static", *objs],
         "linking libsnapkv.so", verbose)


def _build_native(force: bool, verbose: bool):
    """The binding's extension: torch is needed for its headers and libraries only."""
    if not force and not _older(NATIVE, [NATIVE_SOURCE] + NATIVE_HEADERS):
        return
    import torch
    from torch.utils import cpp_extension

    cuda_home = os.path.dirname(os.path.dirname(_nvcc()))
    inc = cpp_extension.include_paths() + [os.path.join(cuda_home, "include"), sysconfig.get_paths()["include"]]
    cmd = [shutil.which("g++") or "c++", "-shared", "-fPIC", "-O2", "-std=c++17", "-Wall",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
           *[x for p in inc for x in ("-isystem", p)],
           os.path.join(CSRC, NATIVE_SOURCE), "-o", NATIVE,
           "-L" + os.path.join(os.path.dirname(torch.__file__), "lib"),
           "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda", "-ltorch", "-ltorch_python"]
    _run(cmd, "g++ " + NATIVE_SOURCE, verbose)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile whatever is out of date; returns the library's path."""
    _build_lib(force, verbose)
    _build_native(force, verbose)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
