"""Builds the sm_103a shared library ``_lib/libmw_bca.so`` in-tree with nvcc.

Each translation unit compiles in parallel, then one nvcc link makes the
shared library against the shared CUDA runtime (found through an rpath to
the toolkit; inside a PyTorch process the runtime PyTorch already loaded is
used).  Beside it ``_lib/_mw_torch.so``, the native half of the Python binding,
with the host compiler against PyTorch's headers.  The driver is reached at run time through the runtime's entry-point
query, so the library loads on machines without a GPU.  A stamp of the sources' hash skips unchanged rebuilds.
"""
from __future__ import annotations

import concurrent.futures as cf
import hashlib
import os
import shutil
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD_DIR = os.path.join(PKG, "_build")
LIB_DIR = os.path.join(PKG, "_lib")
LIB_PATH = os.path.join(LIB_DIR, "libmw_bca.so")
TORCH_SOURCE = "mw_torch.cpp"
TORCH_LIB_PATH = os.path.join(LIB_DIR, "_mw_torch.so")

SOURCES = ["mw_abi.cu", "mw_fwd.cu", "mw_bwd.cu", "mw_commit.cu", "mw_qkv.cu"]
HEADERS = ["mw_ptx.cuh", "mw_internal.h"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
CFLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall",
          "-I" + INCLUDE, "--expt-relaxed-constexpr"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA extension cannot be built")


def _torch_module() -> list:
    """Command that compiles the native half of the Python binding."""
    import torch
    root = os.path.dirname(torch.__file__)
    lib = os.path.join(root, "lib")
    return [shutil.which("g++") or "g++", "-O2", "-std=c++17", "-fPIC", "-shared",
            f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
            f'-DMW_TORCH_VERSION="{torch.__version__}"',
            "-I" + INCLUDE, "-isystem", os.path.join(root, "include"),
            "-isystem", sysconfig.get_paths()["include"],
            "-isystem", os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include"),
            os.path.join(CSRC, TORCH_SOURCE), "-o", TORCH_LIB_PATH + ".tmp",
            "-L" + lib, "-Wl,-rpath," + lib, "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]


def build_torch_module(force: bool = False) -> None:
    """Compile _mw_torch.so if its sources, PyTorch or Python changed.  The
    package works without it (the Python binding's own checks then run on
    every call), so a failure is reported and the build goes on."""
    stamp = os.path.join(BUILD_DIR, "stamp_torch")
    try:
        import torch
        h = hashlib.sha256(f"{torch.__version__} {sys.version}".encode())
        for path in (os.path.join(CSRC, TORCH_SOURCE), os.path.join(INCLUDE, "mw_bca.h")):
            with open(path, "rb") as f:
                h.update(f.read())
        if not force and os.path.exists(TORCH_LIB_PATH) and os.path.exists(stamp):
            with open(stamp) as f:
                if f.read().strip() == h.hexdigest():
                    return
        r = subprocess.run(_torch_module(), capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(r.stdout + r.stderr)
        os.replace(TORCH_LIB_PATH + ".tmp", TORCH_LIB_PATH)
        with open(stamp, "w") as f:
            f.write(h.hexdigest())
    except Exception as e:  # noqa: BLE001
        if os.path.exists(TORCH_LIB_PATH):
            os.remove(TORCH_LIB_PATH)  # never one of other sources
        sys.stderr.write(f"{TORCH_SOURCE}: not built, calls take the longer way: {e}\n")


def _digest() -> str:
    h = hashlib.sha256()
    for name in SOURCES + HEADERS:
        with open(os.path.join(CSRC, name), "rb") as f:
            h.update(name.encode() + f.read())
    with open(os.path.join(INCLUDE, "mw_bca.h"), "rb") as f:
        h.update(f.read())
    # flags without the include directory, so that the digest names the same
    # build on every machine (the checkout path differs)
    h.update(" ".join(ARCH + [f for f in CFLAGS if not f.startswith("-I")]).encode())
    return h.hexdigest()


def build(verbose: bool = False, force: bool = False, ptxas_info: bool = False) -> str:
    """Compile the library if its sources changed; returns the .so path."""
    os.makedirs(BUILD_DIR, exist_ok=True)
    os.makedirs(LIB_DIR, exist_ok=True)
    with cf.ThreadPoolExecutor(max_workers=1) as ex:
        native = ex.submit(build_torch_module, force)
        path = _build_library(verbose, force, ptxas_info)
        native.result()
    return path


def _build_library(verbose: bool, force: bool, ptxas_info: bool) -> str:
    stamp = os.path.join(BUILD_DIR, "stamp")
    digest = _digest()
    if not force and os.path.exists(LIB_PATH) and os.path.exists(stamp):
        with open(stamp) as f:
            if f.read().strip() == digest:
                return LIB_PATH
    nvcc = _nvcc()
    extra = ["-Xptxas", "-v"] if ptxas_info else []

    def compile_one(src: str) -> str:
        obj = os.path.join(BUILD_DIR, src.replace(".cu", ".o"))
        cmd = [nvcc, *ARCH, *CFLAGS, *extra, "-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        if verbose or ptxas_info:
            sys.stderr.write(r.stdout + r.stderr)
        return obj

    with cf.ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = LIB_PATH + ".tmp"
    # shared CUDA runtime: inside a PyTorch process the already-loaded
    # libcudart.so.13 is reused, so the library and PyTorch see one runtime
    # (one current device, one view of stream capture)
    cudart_dir = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "lib64")
    cmd = [nvcc, *ARCH, "-shared", "-cudart", "shared", "-Xlinker", "-rpath=" + cudart_dir,
           "-o", tmp, *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB_PATH)
    with open(stamp, "w") as f:
        f.write(digest)
    return LIB_PATH


if __name__ == "__main__":
    print(build(verbose=True, force="--force" in sys.argv, ptxas_info="--ptxas" in sys.argv))
