"""A handle's memory is filled on the handle's stream.

The allocator hands memory out for that stream: what used it before may still run
there, so a copy on another stream could land too early, and a non-blocking stream
waits for no copy elsewhere.  The CUDA runtime is replaced by a recording one.
"""
import os
import subprocess
import sys

import pytest

import paper_2306_14887_gb300 as tn
from paper_2306_14887_gb300 import build as B

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#include <cuda_runtime_api.h>
#include <stdlib.h>
#include <string.h>
static int own, other;
static void seen(cudaStream_t s) { if (s == (cudaStream_t)64) ++own; else ++other; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(struct cudaDeviceProp* p, int d) {
  memset(p, 0, sizeof *p);
  p->major = 10;
  p->minor = 3;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) { *v = 152; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v) { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { *p = aligned_alloc(256, (n + 255) / 256 * 256); return cudaSuccess; }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned f) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, enum cudaMemcpyKind k) {
  seen(0);
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind k, cudaStream_t st) {
  seen(st);
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) { seen(0); memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) {
  seen(st);
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
int fake_own(void) { return own; }
int fake_other(void) { return other; }
"""

CREATE = r"""
import ctypes as C, sys
import paper_2306_14887_gb300 as tn
fake = C.CDLL(sys.argv[1])
star = [(0, 1), (0, 3), (0, 5), (1, 2), (3, 4), (5, 6)]
edges = star + [(a + 7, b + 7) for a, b in star]  # two components
s = tn.TNState(14, edges, chi=int(sys.argv[2]), prec=sys.argv[3], stream=64, torch_allocator=False)
print(fake.fake_own(), fake.fake_other())
s.close()
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    B.build()
    d = tmp_path_factory.mktemp("fake")
    src, so = d / "fake.c", d / "libfake.so"
    src.write_text(FAKE)
    home = os.path.dirname(os.path.dirname(B.nvcc()))
    subprocess.run(["gcc", "-shared", "-fPIC", "-I", os.path.join(home, "include"), "-o", str(so),
                    str(src)], check=True)
    return str(so)


@pytest.mark.parametrize("chi,prec", [(8, "fp32"), (23, "tf32x3"), (40, "fp32"), (16, "tf32")])
def test_creation_fills_memory_on_the_stream_of_the_handle(fake, chi, prec):
    r = subprocess.run([sys.executable, "-c", CREATE, fake, str(chi), prec], cwd=ROOT,
                       env=dict(os.environ, LD_PRELOAD=fake), capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    own, other = map(int, r.stdout.split())
    assert own > 10 and other == 0
