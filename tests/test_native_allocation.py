"""The native half of the Python binding allocates its outputs without the
interpreter lock: an allocation can wait for the device, and the device for a
callback that needs the lock."""
import os
import subprocess
import sys
import textwrap

import pytest

from paper_2608_01127_gb300 import _build

pytestmark = pytest.mark.gpu

ALLOCATOR = r"""
#include <Python.h>
#include <cuda_runtime.h>
#include <atomic>
extern "C" {
static std::atomic<int> with_lock{0}, without{0};
void* test_malloc(ssize_t size, int, cudaStream_t) {
  ++(PyGILState_Check() ? with_lock : without);
  void* p = nullptr;
  return cudaMalloc(&p, size > 0 ? size : 1) == cudaSuccess ? p : nullptr;
}
void test_free(void* p, ssize_t, int, cudaStream_t) { cudaFree(p); }
int allocations(int locked) { return (locked ? with_lock : without).exchange(0); }
}
"""

CALLS = """
    import ctypes, sys, torch
    sys.path.insert(0, {root!r})
    torch.cuda.memory.change_current_allocator(
        torch.cuda.memory.CUDAPluggableAllocator({lib!r}, "test_malloc", "test_free"))
    import paper_2608_01127_gb300 as mw
    mw.library()
    count = ctypes.CDLL({lib!r}).allocations
    g = torch.Generator("cuda").manual_seed(1)
    bf = lambda *s: torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16)
    q, k, v, do = (bf(1, 2, 128, 64) for _ in range(4))
    kc, vc = bf(1, 2, 2048, 64), bf(1, 2, 2048, 64)
    o, lse = mw.mw_bca_fwd(q, k, v, 64)
    for name, call, n in (
            ("fwd", lambda: mw.mw_bca_fwd(q, k, v, 64), 2),
            ("bwd", lambda: mw.mw_bca_bwd(q, k, v, o, lse, do, 64), 4),
            ("cache", lambda: mw.mw_bca_cache_fwd(q, k, v, kc, vc, 0, 2048, 64), 3),
            ("step", lambda: mw.mw_bca_cache_step(q, k, v, kc, vc, 0, 2048, 0, 64, 64), 3),
            ("qkv", lambda: mw.mw_qkv_rope_split(bf5), 3)):
        bf5 = bf(1, 50, 3, 2, 64)
        count(0), count(1)
        out = call()
        print(name, n, count(0), count(1))
    torch.cuda.synchronize()
"""


def test_outputs_are_allocated_without_the_lock(tmp_path):
    source, lib = tmp_path / "allocator.cpp", tmp_path / "allocator.so"
    source.write_text(ALLOCATOR)
    cuda = os.path.dirname(os.path.dirname(_build._nvcc()))
    import sysconfig
    subprocess.run(["g++", "-shared", "-fPIC", "-I" + sysconfig.get_paths()["include"], "-I" + cuda + "/include",
                    str(source), "-o", str(lib), "-L" + cuda + "/lib64", "-lcudart"], check=True, capture_output=True)
    code = textwrap.dedent(CALLS.format(root=_build.ROOT, lib=str(lib)))
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = [line.split() for line in r.stdout.splitlines()]
    assert [line[0] for line in lines] == ["fwd", "bwd", "cache", "step", "qkv"]
    for name, expected, without, locked in lines:
        assert (int(without), int(locked)) == (int(expected), 0), name
