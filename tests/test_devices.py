"""Kernel attributes belong to a function on one device: the library's launches
on a second device, against a CUDA runtime that answers for two devices and
refuses, as the real one does, a launch with more shared memory than the
function may have on the current device."""
import os
import shutil
import subprocess
import sys
import textwrap

import pytest

from paper_2608_01127_gb300 import _build

RUNTIME = r"""
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <map>
#include <utility>
static int device = 0, registers = 0, launches = 0;
static cudaError_t last = cudaSuccess;
static std::map<std::pair<int, const void*>, int> shared_memory;
static CUresult encode(...) { return CUDA_SUCCESS; }
static cudaError_t launch(const void* f, size_t bytes) {
  const auto it = shared_memory.find({device, f});
  const size_t limit = it == shared_memory.end() ? 49152 : it->second;
  if (bytes > limit) return last = cudaErrorInvalidValue;
  ++launches;
  return cudaSuccess;
}
extern "C" {
void fake(int dev, int regs) { device = dev; registers = regs; }
int fake_launches() { int n = launches; launches = 0; return n; }
cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { device = d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = (void*)0x100000; return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** p, unsigned, unsigned long long,
                                             enum cudaDriverEntryPointQueryResult* r) {
  *p = (void*)encode;
  *r = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(struct cudaFuncAttributes* a, const void*) {
  *a = cudaFuncAttributes{};
  a->numRegs = registers;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute, int v) {
  shared_memory[{device, f}] = v;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return launch(f, c->dynamicSmemBytes);
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t bytes, cudaStream_t) {
  return launch((const void*)k, bytes);
}
cudaError_t cudaGetLastError() { cudaError_t e = last; last = cudaSuccess; return e; }
}
"""

CALLS = """
    import ctypes, sys
    fake, lib = ctypes.CDLL({fake!r}), ctypes.CDLL({lib!r})
    lib.mw_last_error.restype = ctypes.c_char_p
    lib.mw_bca_bwd_workspace_size.restype = ctypes.c_size_t
    P = ctypes.c_void_p(0x10000)
    F, Z = ctypes.c_float, ctypes.c_size_t
    for d in (64, 72, 128):
        for device in (0, 1, 0, 1):
            fake.fake(device, 168)
            code = lib.mw_bca_fwd(P, P, P, P, P, 1, 2, 2, 64, d, F(0.125), None)
            print("fwd", d, device, code, fake.fake_launches(), lib.mw_last_error().decode())
            fake.fake(device, 128)
            ws = lib.mw_bca_bwd_workspace_size(1, 2, 2, 64, d)
            code = lib.mw_bca_bwd(P, P, P, P, P, P, P, P, P, P, Z(ws), 1, 2, 2, 64, d, F(0.125), None)
            print("bwd", d, device, code, fake.fake_launches(), lib.mw_last_error().decode())
    # a launch register count that the kernels' split does not fit is refused, on each device anew
    for device in (2, 3):
        fake.fake(device, 100)
        code = lib.mw_bca_fwd(P, P, P, P, P, 1, 2, 2, 64, 64, F(0.125), None)
        print("refused", 64, device, int(code == 0), fake.fake_launches())
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_two_devices(tmp_path):
    lib = _build.build()
    source, fake = tmp_path / "runtime.cpp", tmp_path / "runtime.so"
    source.write_text(RUNTIME)
    cuda = os.path.dirname(os.path.dirname(_build._nvcc()))
    subprocess.run(["g++", "-shared", "-fPIC", "-I" + cuda + "/include", str(source), "-o", str(fake)],
                   check=True, capture_output=True)
    code = textwrap.dedent(CALLS.format(fake=str(fake), lib=lib))
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True,
                       env={**os.environ, "LD_PRELOAD": str(fake)})
    assert r.returncode == 0, r.stderr[-2000:]
    lines = [line.split() for line in r.stdout.splitlines()]
    assert len(lines) == 26
    for what, d, device, code, launches, *message in lines:
        expected = {"fwd": "1", "bwd": "3", "refused": "0"}[what]
        assert (code, launches) == ("0", expected), (what, d, device, message)
