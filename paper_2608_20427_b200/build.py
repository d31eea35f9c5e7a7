"""Builds libbf1.so (the C-ABI library, nvcc for sm_100a) and the extension module _host (the binding's call path, g++) in-tree."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libbf1.so")
HOST_SOURCE = os.path.join(CSRC, "bf1_host.cpp")
SOURCES = ["bf1_plan.cu", "bf1_attn.cu", "bf1_noalloc.cu", "bf1_decode.cu", "bf1_bwd.cu", "bf1_shard.cu"]
HEADERS = ["bf1_common.cuh", os.path.join("..", "..", "include", "bf1.h")]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def is_stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, s) for s in SOURCES + HEADERS]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, out: str = None, defines=()) -> str:
    """Compile the library if it is missing or older than its sources; return its path.
    `out` / `defines` compile a variant of the sources to another path (the binding never loads it)."""
    if out is None and not force and not is_stale():
        return LIB
    lib = out or LIB
    tmp = lib + ".tmp.%d" % os.getpid()
    cmd = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
           "-Xcompiler", "-fPIC", "-shared", "-o", tmp]
    cmd += ["-D" + d for d in defines]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, s) for s in SOURCES]
    res = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed building libbf1.so:\n" + res.stdout)
    os.replace(tmp, lib)
    return lib


def host_path() -> str:
    """The extension module is compiled against the C++ ABI of one torch and one Python, which its name says: with another of
    either it is another file."""
    import torch
    return os.path.join(HERE, "_host.%s-torch%s.so" % (sys.implementation.cache_tag, torch.__version__))


def build_host(force: bool = False) -> str:
    """Compile the extension module that marshals torch tensors into the C ABI, if there is none for this torch and Python or it
    is older than its source; return its path.  It links libbf1.so from its own folder, which has to be there already."""
    deps = [HOST_SOURCE, os.path.join(CSRC, HEADERS[1])]
    host = host_path()
    if not force and os.path.exists(host) and all(os.path.getmtime(d) <= os.path.getmtime(host) for d in deps):
        return host
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.path.join(os.path.dirname(os.path.dirname(_nvcc())) or "/usr/local/cuda", "include")
    tmp = host + ".tmp.%d" % os.getpid()
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch._C._GLIBCXX_USE_CXX11_ABI,
           "-I" + sysconfig.get_paths()["include"], "-I" + os.path.join(root, "include"),
           "-I" + os.path.join(root, "include", "torch", "csrc", "api", "include"), "-I" + cuda, HOST_SOURCE, "-o", tmp,
           "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda",
           "-L" + HERE, "-l:" + os.path.basename(LIB), "-Wl,-rpath,$ORIGIN"]
    res = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if res.returncode != 0:
        raise RuntimeError("g++ failed building _host:\n" + res.stdout)
    os.replace(tmp, host)
    return host


if __name__ == "__main__":
    print(build(force=True, verbose=True))
    print(build_host(force=True))
