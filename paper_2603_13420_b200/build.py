"""Build libpskv.so in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the Python face _native.so with g++.

    python -m paper_2603_13420_b200.build [--force] [--verbose]
"""
from __future__ import annotations

import os
import subprocess
import sys

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG_DIR)
CSRC = os.path.join(PKG_DIR, "csrc")
INCLUDE = os.path.join(ROOT, "include")
LIB_PATH = os.path.join(PKG_DIR, "libpskv.so")
NATIVE_SRC = os.path.join(CSRC, "pskv_python.cpp")
NATIVE_PATH = os.path.join(PKG_DIR, "_native.so")

SOURCES = ["pskv_api.cu", "pskv_simt.cu", "pskv_tc_fwd.cu", "pskv_tc_fwd_pair.cu", "pskv_tc_bwd.cu", "pskv_tc_bwd_prefix.cu", "pskv_noalloc.cu", "pskv_selftest.cu", "pskv_ce.cu"]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _deps():
    deps = [os.path.join(INCLUDE, "pskv.h")]
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh", ".h")):
            deps.append(os.path.join(CSRC, name))
    return deps


def _older(target, sources) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(p) > os.path.getmtime(target) for p in sources)


def _torch_dir() -> str:
    import importlib.util

    return os.path.dirname(importlib.util.find_spec("torch").origin)


def built_for() -> str:
    """The interpreter and torch that the extension module is built for (torch itself need not be imported)."""
    version = {}
    with open(os.path.join(_torch_dir(), "version.py")) as f:
        exec(f.read(), version)
    return "%s torch %s" % (sys.implementation.cache_tag, version["__version__"])


def _native_stale() -> bool:
    if _older(NATIVE_PATH, [NATIVE_SRC, _deps()[0]]):
        return True
    with open(NATIVE_PATH, "rb") as f:
        return built_for().encode() + b"\0" not in f.read()


def is_stale() -> bool:
    return _older(LIB_PATH, _deps()) or _native_stale()


def _build_native() -> None:
    """The Python extension module; it needs torch's headers and libraries, not CUDA kernels."""
    import sysconfig

    torch_dir = _torch_dir()
    inc = os.path.join(torch_dir, "include")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    tmp = NATIVE_PATH + ".tmp.%d" % os.getpid()
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", '-DPSKV_BUILT_FOR="%s"' % built_for(), "-I", INCLUDE, "-I", inc,
                    "-I", os.path.join(inc, "torch", "csrc", "api", "include"), "-I", sysconfig.get_paths()["include"],
                    "-I", os.path.join(cuda, "include"), NATIVE_SRC, "-o", tmp, "-L", os.path.join(torch_dir, "lib"),
                    "-ltorch_python", "-ltorch", "-ltorch_cpu", "-ltorch_cuda", "-lc10", "-lc10_cuda"], check=True)
    os.replace(tmp, NATIVE_PATH)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every CUDA source into paper_2603_13420_b200/libpskv.so, and the extension module beside it; returns the
    library's path."""
    if force or _native_stale():
        _build_native()
    if not force and not _older(LIB_PATH, _deps()):
        return LIB_PATH
    objs = []
    procs = []
    for src in SOURCES:
        obj = os.path.join(CSRC, src[:-3] + ".o")
        cmd = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3",
               "-std=c++17", "--use_fast_math", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC,
               "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT,
                                            text=True)))
        objs.append(obj)
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write("[%s]\n%s\n" % (src, out))
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = LIB_PATH + ".tmp.%d" % os.getpid()
    subprocess.run([_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", tmp]
                   + objs + ["-cudart", "static"], check=True)
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
