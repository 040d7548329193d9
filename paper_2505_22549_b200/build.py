"""Builds libdesloc.so (sm_100a) in-tree with nvcc; no JIT cache, no torch extension.

    python -m paper_2505_22549_b200.build [--force] [--verbose]

Translation units compile in parallel; the results are paper_2505_22549_b200/lib/libdesloc.so and, built with g++
against torch's headers, the CPython module paper_2505_22549_b200/_native.so that module.py calls the library through.
"""
from __future__ import annotations

import concurrent.futures as cf
import glob
import hashlib
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "build")
LIBDIR = os.path.join(HERE, "lib")
LIB = os.path.join(LIBDIR, "libdesloc.so")
NATIVE_SRC = os.path.join(CSRC, "desloc_py.cpp")
NATIVE = os.path.join(HERE, "_native.so")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden", "--threads", "2",
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    raise RuntimeError("nvcc not found")


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _fingerprint(src: str) -> str:
    """Hash of one translation unit with every header it may include and the flags."""
    h = hashlib.sha256()
    files = [src] + sorted(glob.glob(os.path.join(CSRC, "*.cuh"))) + \
        sorted(glob.glob(os.path.join(INCLUDE, "*.h")))
    for f in files:
        h.update(os.path.basename(f).encode())
        h.update(open(f, "rb").read())
    h.update(" ".join(NVCC_FLAGS).encode())
    return h.hexdigest()


def _build_native(force: bool) -> None:
    """The CPython module (host code only)."""
    import sysconfig
    import torch
    from torch.utils import cpp_extension as ce
    libs = os.path.join(os.path.dirname(torch.__file__), "lib")
    dirs = ce.include_paths() + [sysconfig.get_paths()["include"], os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include")]
    tmp, stamp = NATIVE + f".tmp{os.getpid()}", os.path.join(OBJ, "_native.stamp")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
           f'-DDESLOC_TORCH_VERSION="{torch.__version__}"']
    cmd += [a for d in dirs for a in ("-isystem", d)] + [NATIVE_SRC, "-L", libs]
    cmd += ["-ltorch_python", "-ltorch_cpu", "-ltorch", "-lc10_cuda", "-lc10"]
    h = hashlib.sha256(" ".join(cmd + [torch.__version__, sys.version]).encode())
    for f in [NATIVE_SRC] + sorted(glob.glob(os.path.join(INCLUDE, "*.h"))):
        h.update(open(f, "rb").read())
    if not force and os.path.exists(NATIVE) and os.path.exists(stamp) and open(stamp).read() == h.hexdigest():
        return
    r = subprocess.run(cmd + ["-o", tmp], capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed on {NATIVE_SRC}:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, NATIVE)
    with open(stamp, "w") as f:
        f.write(h.hexdigest())


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every translation unit (in parallel) and link the shared library.
    verbose passes -Xptxas -v and prints the compiler's register / spill report to stderr."""
    return _build(force, verbose, [])


def _build(force: bool, verbose: bool, extra_flags) -> str:
    os.makedirs(OBJ, exist_ok=True)
    os.makedirs(os.path.dirname(LIB), exist_ok=True)
    nvcc = _nvcc()
    flags = NVCC_FLAGS + extra_flags + (["-Xptxas", "-v"] if verbose else [])

    def compile_one(src):
        obj = os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")
        stamp = obj + ".stamp"
        fp = _fingerprint(src) + " ".join(extra_flags)
        if (not force and os.path.exists(obj) and os.path.exists(stamp)
                and open(stamp).read() == fp):
            return obj, False
        cmd = [nvcc] + flags + ["-I", INCLUDE, "-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        if verbose:
            sys.stderr.write(r.stderr)
        with open(stamp, "w") as f:
            f.write(fp)
        return obj, True

    with cf.ThreadPoolExecutor(max_workers=min(8, os.cpu_count() or 2)) as ex:
        native = ex.submit(_build_native, force)
        results = list(ex.map(compile_one, _sources()))
        native.result()
    objs = [o for o, _ in results]
    if not any(changed for _, changed in results) and os.path.exists(LIB):
        return LIB
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", tmp] + objs + ["-ldl"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
