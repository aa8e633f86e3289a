"""Builds libkvs.so (the C-ABI library, nvcc for sm_100a) and the extension module _kvs_native (the native calls of the binding, g++) in-tree.

    python -m paper_2609_35750_b200.build [--force]
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
LIB = os.path.join(HERE, "libkvs.so")
NATIVE_SOURCE = os.path.join(CSRC, "kvs_native.cpp")
SOURCES = ["kvs_api.cu", "kvs_meta.cu", "kvs_fwd.cu", "kvs_fwd_dual.cu", "kvs_bwd.cu", "kvs_bwd_pair.cu", "kvs_bwd_noalloc.cu", "kvs_decode.cu", "kvs_rope.cu"]
HEADERS = [os.path.join(CSRC, "kvs_common.cuh"), os.path.join(CSRC, "kvs_bwd.cuh"), os.path.join(INCLUDE, "kvs.h")]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I" + INCLUDE, "-I" + CSRC]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def native_path() -> str:
    """The module depends on Python's and torch's binary interface: both versions are in its name, so that one compiled against
    others is neither up to date nor loaded."""
    import torch
    return os.path.join(HERE, f"_kvs_native-{torch.__version__}{sysconfig.get_config_var('EXT_SUFFIX')}")


def native_command() -> list:
    import torch
    from torch.utils.cpp_extension import include_paths, library_paths
    cuda = os.path.dirname(os.path.dirname(_nvcc())) if os.path.sep in _nvcc() else "/usr/local/cuda"
    dirs = include_paths() + [sysconfig.get_paths()["include"], os.path.join(cuda, "include"), INCLUDE]
    return (["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch.compiled_with_cxx11_abi()] +
            ["-I" + d for d in dirs] + [NATIVE_SOURCE, "-o", native_path()] + ["-L" + d for d in library_paths()] +
            ["-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"])


def _older(target: str, deps: list) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in deps)


def needs_build() -> bool:
    return (_older(LIB, [os.path.join(CSRC, s) for s in SOURCES] + HEADERS) or
            _older(native_path(), [NATIVE_SOURCE, os.path.join(INCLUDE, "kvs.h")]))


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    objdir = os.path.join(HERE, "build")
    os.makedirs(objdir, exist_ok=True)
    nvcc = _nvcc()
    procs = []
    for s in SOURCES:
        obj = os.path.join(objdir, s.replace(".cu", ".o"))
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", os.path.join(CSRC, s), "-o", obj]
        procs.append((s, obj, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    native = subprocess.Popen(native_command(), stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    objs = []
    for s, obj, p in procs:
        out, _ = p.communicate()
        if verbose and out:
            print(out)
        if p.returncode != 0:
            raise RuntimeError(f"nvcc failed on {s}:\n{out}")
        objs.append(obj)
    cmd = [nvcc, "-shared", "-o", LIB] + objs
    r = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}")
    out, _ = native.communicate()
    if native.returncode != 0:
        raise RuntimeError(f"g++ failed on {os.path.basename(NATIVE_SOURCE)}:\n{out}")
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
