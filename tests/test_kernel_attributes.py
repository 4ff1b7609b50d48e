"""Contexts on different threads do not disturb each other through kernel attributes.
The dynamic shared memory limit of a kernel belongs to the device, not to a call: were
it set to a call's own size, a small call between a large call's setting and its launch
would make that launch fail.  So every call must set the same limit, and no launch may
exceed it.

Host test: the library's calls run against a stand-in for the CUDA runtime (preloaded;
it starts nothing) that records the limits set and the launches."""

import collections
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUNTIME = r"""
#include <cuda_runtime_api.h>
#include <cstdio>
#include <cstdlib>
#include <cstring>
static FILE *out() { static FILE *f = fopen(getenv("ATTR_LOG"), "w"); return f; }
extern "C" {
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) { fprintf(out(), "limit %p %d\n", f, v); fflush(out()); }
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) {
  fprintf(out(), "launch %p %zu\n", f, c->dynamicSmemBytes); fflush(out());
  return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int) {
  memset(p, 0, sizeof *p);
  p->multiProcessorCount = 152;
  p->sharedMemPerBlockOptin = 232448;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 0;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
  *n = 4;
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
  memset(a, 0, sizeof *a);
  a->type = cudaMemoryTypeDevice;
  a->devicePointer = const_cast<void *>(p);
  return cudaSuccess;
}
cudaError_t cudaMalloc(void **p, size_t) { static char *next = (char *)0x10000000; *p = next; next += 0x10000; return cudaSuccess; }
cudaError_t cudaMallocHost(void **p, size_t n) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFree(void *) { return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaHostGetDevicePointer(void **d, void *p, unsigned) { *d = p; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)1; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
}
"""

CALLS = r"""
import ctypes, importlib.util, sys
spec = importlib.util.spec_from_file_location("native", sys.argv[1])
N = importlib.util.module_from_spec(spec)
spec.loader.exec_module(N)
L = N.lib()
ctx = ctypes.c_void_p()
assert L.denoise_create(ctypes.byref(ctx), 0, 2_000_000, 1) == 0
assert L.denoise_set_cross_leaf(ctx, 1) == 0
for train in (0, 1):
    assert L.denoise_set_training(ctx, train) == 0
    for n in (300, 1500, 5000, 36750, 700_000, 2_000_000):
        for cap in (30, 64, 128, 256, 512, 1024, 2048, 0xFFFFFFFF):
            for k in (8, 16, 32, 64):
                for cross in (0, 1):
                    p = N.denoise_params(k, cap, 21, 3.0, 4, 0.2, 1.0, 1.0, 2.0, 1e-12, 1e-12, 0, 0.95, 0.0, 0.05, 0, 0, cross)
                    assert L.denoise_run(ctx, 0x7000, n, ctypes.byref(p), 0x8000, 0x9000, 0xA000, None) == 0
"""


def test_every_call_sets_the_same_limits(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not available")
    from paper_2512_10386_gb300 import _native, build
    build.build()
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    src, so, log = tmp_path / "runtime.cpp", tmp_path / "runtime.so", tmp_path / "log"
    src.write_text(RUNTIME)
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I", inc, str(src), "-o", str(so)], check=True)
    r = subprocess.run([sys.executable, "-c", CALLS, _native.LIB_PATH.replace("libgravdenoise.so", "_native.py")],
                       capture_output=True, text=True, env={**os.environ, "LD_PRELOAD": str(so), "ATTR_LOG": str(log)})
    assert r.returncode == 0, r.stderr
    limits, launches = collections.defaultdict(set), collections.defaultdict(int)
    for line in log.read_text().splitlines():
        what, kernel, value = line.split()
        if what == "limit":
            limits[kernel].add(int(value))
        else:
            launches[kernel] = max(launches[kernel], int(value))
    assert len(limits) >= 10 and len(launches) >= 20
    assert all(len(v) == 1 for v in limits.values()), {k: sorted(v) for k, v in limits.items() if len(v) > 1}
    for kernel, largest in launches.items():
        assert largest <= max(limits.get(kernel, {48 << 10})), (kernel, largest)
