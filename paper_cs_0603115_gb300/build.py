"""Build step of libff.so: nvcc for sm_103a, one object per translation unit
compiled in parallel, then one shared-library link; and of _ffnative.so, the
native front of the Python wrappers (one C++ file against torch's headers),
beside it.  In-tree: the libraries land next to this file, the objects under
``_build/``.

Flags that the float-float arithmetic relies on:
  -fmad=false           no contraction of a*b + c into an FMA anywhere
                        (the operators use explicit _rn intrinsics as well);
  -ftz=false            binary32 subnormals are kept;
  -prec-div/-prec-sqrt  IEEE round-to-nearest division and square root.
"""
from __future__ import annotations

import concurrent.futures as cf
import hashlib
import os
import shutil
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD_DIR = os.path.join(ROOT, "_build")
LIB_NAME = "libff.so"
LIB_PATH = os.path.join(HERE, LIB_NAME)
NATIVE_SRC = os.path.join(CSRC, "ff_torch.cpp")
NATIVE_PATH = os.path.join(HERE, "_ffnative.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-fmad=false", "-ftz=false", "-prec-div=true",
              "-prec-sqrt=true", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
              "--expt-relaxed-constexpr"]


def nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libff.so")


def sources() -> list[str]:
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _inputs() -> list[str]:
    files = sources() + [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cuh")]
    files.append(os.path.join(ROOT, "include", "ff.h"))
    return sorted(files)


def build_id() -> str:
    h = hashlib.sha256()
    for f in _inputs():
        with open(f, "rb") as fh:
            h.update(os.path.basename(f).encode())
            h.update(fh.read())
    h.update(" ".join(ARCH + NVCC_FLAGS).encode())
    return h.hexdigest()[:16]


def _compile(src: str, bid: str, extra: list[str]) -> str:
    obj = os.path.join(BUILD_DIR, os.path.basename(src)[:-3] + ".o")
    cmd = [nvcc(), *ARCH, *NVCC_FLAGS, *extra, f'-DFF_BUILD_ID="{bid}"', "-c", src, "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
    if "-v" in extra and r.stderr:
        print(r.stderr)
    return obj


def _native_command(out: str) -> list[str]:
    import sysconfig

    import torch
    root = os.path.dirname(torch.__file__)
    lib = os.path.join(root, "lib")
    cuda = os.path.dirname(os.path.dirname(nvcc()))
    return ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
            f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
            *[f"-I{d}" for d in (os.path.join(root, "include"), sysconfig.get_paths()["include"],
                                 os.path.join(cuda, "include"))],
            NATIVE_SRC, "-o", out, f"-L{lib}", "-ltorch_python", "-ltorch_cpu", "-lc10_cuda", "-lc10", f"-Wl,-rpath,{lib}"]


def build_native(force: bool = False) -> str:
    """Compile _ffnative.so if its source, ff.h, torch or the command changed."""
    import torch
    h = hashlib.sha256(torch.__version__.encode())
    for f in (NATIVE_SRC, os.path.join(ROOT, "include", "ff.h")):
        with open(f, "rb") as fh:
            h.update(fh.read())
    h.update(" ".join(_native_command(NATIVE_PATH)).encode())
    bid = h.hexdigest()[:16]
    stamp = os.path.join(BUILD_DIR, "native_id")
    if not force and os.path.exists(NATIVE_PATH) and os.path.exists(stamp) and open(stamp).read().strip() == bid:
        return NATIVE_PATH
    os.makedirs(BUILD_DIR, exist_ok=True)
    tmp = NATIVE_PATH + f".tmp{os.getpid()}"
    r = subprocess.run(_native_command(tmp), capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed for {NATIVE_SRC}:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, NATIVE_PATH)
    with open(stamp, "w") as fh:
        fh.write(bid)
    return NATIVE_PATH


def build(force: bool = False, verbose: bool = False, extra: list[str] | None = None) -> str:
    """Compile libff.so and _ffnative.so if any of their inputs changed; returns
    the path of libff.so."""
    with cf.ThreadPoolExecutor(max_workers=1) as ex:
        native = ex.submit(build_native, force)
        path = _build_library(force, verbose, extra)
        native.result()
    return path


def _build_library(force: bool, verbose: bool, extra: list[str] | None) -> str:
    bid = build_id()
    stamp = os.path.join(BUILD_DIR, "build_id")
    if (not force and os.path.exists(LIB_PATH) and os.path.exists(stamp)
            and open(stamp).read().strip() == bid):
        return LIB_PATH
    os.makedirs(BUILD_DIR, exist_ok=True)
    extra = list(extra or [])
    if verbose:
        extra += ["-Xptxas", "-v"]
    srcs = sources()
    with cf.ThreadPoolExecutor(max_workers=min(len(srcs), os.cpu_count() or 4)) as ex:
        objs = list(ex.map(lambda s: _compile(s, bid, extra), srcs))
    tmp = LIB_PATH + f".tmp{os.getpid()}"
    cmd = [nvcc(), *ARCH, "-shared", "-cudart", "shared", "-o", tmp, *objs,
           "-Xlinker", "-rpath,/usr/local/cuda/lib64"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB_PATH)
    with open(stamp, "w") as fh:
        fh.write(bid)
    return LIB_PATH


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
