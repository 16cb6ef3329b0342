"""Builds ``libsdgp.so`` (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and ``_sdgp_torch.so``, the module
that calls it with torch tensors (plain C++ against torch's headers, no device code)."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libsdgp.so")
SOURCES = ["prune.cu", "rank.cu", "dgrad.cu", "dgrad_general.cu", "dgrad_halo_sparse.cu", "dgrad_halo_dense.cu",
           "dgrad_halo_fused.cu", "dgrad_rows.cu", "dgrad_grouped.cu", "api.cu", "static_scratch.cu", "channel.cu", "grouped.cu"]
BINDING = os.path.join(HERE, "_sdgp_torch.so")
BINDING_SOURCES = [os.path.join(CSRC, f) for f in ("torch_binding.cpp", "torch_autograd.cpp")]
HEADERS = ["ptx.cuh", "sdgp_internal.cuh", "prune_core.cuh", "dgrad_common.cuh", "dgrad_general.cuh", "dgrad_halo.cuh",
           "dgrad_halo_params.cuh", "dgrad_prune.cuh", "dgrad_rows.cuh", os.path.join("..", "..", "include", "sdgp.h")]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _stale(target, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def needs_build() -> bool:
    return _stale(LIB, [os.path.join(CSRC, f) for f in SOURCES + HEADERS] + [os.path.abspath(__file__)])


def build_binding(force: bool = False) -> str:
    """The torch module; needs ``libsdgp.so`` beside it (it finds it through its run path)."""
    if not force and not _stale(BINDING, BINDING_SOURCES + [os.path.join(CSRC, "torch_autograd.h"), os.path.join(CSRC, "sdgp_internal.cuh"),
                                                            os.path.join(HERE, "..", "include", "sdgp.h"), os.path.abspath(__file__)]):
        return BINDING
    from torch.utils import cpp_extension
    tmp = BINDING + ".%d.tmp" % os.getpid()
    include = [sysconfig.get_paths()["include"]] + cpp_extension.include_paths("cuda")
    libs = cpp_extension.library_paths("cuda")
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-o", tmp] + BINDING_SOURCES
    cmd += ["-I" + d for d in include] + ["-L" + HERE, "-lsdgp"] + ["-L" + d for d in libs]
    cmd += ["-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch", "-ltorch_python", "-Wl,-rpath,$ORIGIN"]
    subprocess.check_call(cmd)
    os.replace(tmp, BINDING)
    return BINDING


def _compile(src: str, force: bool, verbose: bool) -> str:
    """One translation unit to an object file under ``_build/`` (skipped while it is newer than everything it reads)."""
    obj = os.path.join(HERE, "_build", os.path.splitext(src)[0] + ".o")
    deps = [os.path.join(CSRC, f) for f in [src] + HEADERS] + [os.path.abspath(__file__)]
    if force or _stale(obj, deps):
        tmp = "%s.%d.tmp.o" % (obj, os.getpid())
        cmd = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC"]
        subprocess.check_call(cmd + (["-Xptxas", "-v"] if verbose else []) + ["-c", "-o", tmp, os.path.join(CSRC, src)])
        os.replace(tmp, obj)
    return obj


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    os.makedirs(os.path.join(HERE, "_build"), exist_ok=True)
    with ThreadPoolExecutor() as pool:
        objects = list(pool.map(lambda src: _compile(src, force, verbose), SOURCES))
    tmp = LIB + ".%d.tmp" % os.getpid()
    subprocess.check_call([_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-Xcompiler", "-fPIC", "-o", tmp] + objects)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
    print(build_binding(force="--force" in sys.argv))
