"""Builds the native code in-tree: the CUDA library ``libmsd.so`` (sm_100a only) and the call module ``_native.so`` next
to this file.

Every ``csrc/*.cu`` is compiled to an object of its own (in parallel, and only when it or a header changed), then the
objects are linked into one shared library; ``csrc/native_call.cpp`` marshals torch tensors into its calls.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

_HERE = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_HERE)
LIB_PATH = os.path.join(_HERE, "libmsd.so")
NATIVE_PATH = os.path.join(_HERE, "_native.so")
NATIVE_SRC = os.path.join(_HERE, "csrc", "native_call.cpp")
OBJ_DIR = os.path.join(_HERE, "build")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
    "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
]


def sources():
    return sorted(glob.glob(os.path.join(_HERE, "csrc", "*.cu")))


def _headers():
    return glob.glob(os.path.join(_HERE, "csrc", "*.h")) + glob.glob(os.path.join(_HERE, "csrc", "*.cuh")) + \
        glob.glob(os.path.join(_ROOT, "include", "*.h"))


def needs_build() -> bool:
    return _lib_stale() or _native_stale()


def _lib_stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    t = os.path.getmtime(LIB_PATH)
    return any(os.path.getmtime(d) > t for d in sources() + _headers())


def _native_tag() -> str:
    """What the call module is built for, and carries as a string: torch's binary interface changes with its version."""
    import torch
    return "msd call module for torch %s, python %d.%d" % (torch.__version__, sys.version_info[0], sys.version_info[1])


def _native_stale() -> bool:
    if not os.path.exists(NATIVE_PATH):
        return True
    t = os.path.getmtime(NATIVE_PATH)
    if any(os.path.getmtime(d) > t for d in (NATIVE_SRC, os.path.join(_ROOT, "include", "msd.h"))):
        return True
    with open(NATIVE_PATH, "rb") as f:
        return _native_tag().encode() + b"\0" not in f.read()


def _build_native():
    """The call module: a CPython extension against torch's headers, linked to libmsd.so beside it."""
    import sysconfig
    import torch
    troot = os.path.dirname(torch.__file__)
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++20", "-fPIC", "-shared", "-fvisibility=hidden",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch.compiled_with_cxx11_abi(), '-DMSD_BUILT_FOR="%s"' % _native_tag(), NATIVE_SRC, "-o", NATIVE_PATH,
           "-I", os.path.join(_ROOT, "include"), "-I", sysconfig.get_paths()["include"],
           "-isystem", os.path.join(troot, "include"), "-isystem", os.path.join(troot, "include", "torch", "csrc", "api", "include"),
           "-isystem", os.path.join(os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"))), "include"),
           "-L", _HERE, "-l:libmsd.so", "-Wl,-rpath,$ORIGIN",
           "-L", os.path.join(troot, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("building _native.so failed")


def _obj(src):
    return os.path.join(OBJ_DIR, os.path.basename(src)[:-3] + ".o")


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ and link them into one shared library (nvcc cross-compiles without a GPU)."""
    if not force and not _lib_stale():
        if _native_stale():
            _build_native()
        return LIB_PATH
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    os.makedirs(OBJ_DIR, exist_ok=True)
    hdr_time = max([os.path.getmtime(h) for h in _headers()] + [os.path.getmtime(__file__)])
    base = [nvcc] + NVCC_FLAGS + ["-I", os.path.join(_ROOT, "include"), "-I", os.path.join(_HERE, "csrc")]
    if verbose:
        base += ["-Xptxas", "-v"]

    def compile_one(src):
        obj = _obj(src)
        if not force and os.path.exists(obj) and os.path.getmtime(obj) > max(os.path.getmtime(src), hdr_time):
            return 0, ""
        res = subprocess.run(base + ["-c", src, "-o", obj], capture_output=True, text=True)
        return res.returncode, res.stdout + res.stderr

    srcs = sources()
    with ThreadPoolExecutor(max_workers=min(len(srcs), os.cpu_count() or 4)) as ex:
        results = list(ex.map(compile_one, srcs))
    failed = False
    for (rc, out), src in zip(results, srcs):
        if rc != 0 or (verbose and out):
            sys.stderr.write("== %s\n%s" % (os.path.basename(src), out))
        failed = failed or rc != 0
    if failed:
        raise RuntimeError("nvcc failed")
    link = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-cudart", "static", "-o", LIB_PATH,
            "-Xlinker", "-soname=libmsd.so"] + [_obj(s) for s in srcs]
    res = subprocess.run(link, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("nvcc link failed")
    if force or _native_stale():
        _build_native()
    return LIB_PATH


if __name__ == "__main__":
    build(force="-f" in sys.argv, verbose="-v" in sys.argv)
    print(LIB_PATH)
