"""Kernel attributes are set on every device the library is used on, once each.

An attribute such as the shared-memory limit belongs to one device: a kernel
whose limit was raised on the first device only cannot be launched on a second
one.  The CUDA runtime is replaced by a recording one, so no GPU is needed.
"""
import os
import subprocess
import sys

import pytest

import paper_2306_14887_gb300 as tn
from paper_2306_14887_gb300 import build as B

FAKE = r"""
static int device;
static int count[4];
static unsigned long sum[4];
int cudaGetDevice(int* d) { *d = device; return 0; }
int cudaDeviceGetAttribute(int* v, int attr, int d) { *v = 152; return 0; }
int cudaFuncSetAttribute(const void* f, int attr, int value) {
  ++count[device];
  sum[device] = sum[device] * 1000003u + (unsigned long)f * 31u + attr * 7u + value;
  return 0;
}
void fake_use(int d) { device = d; }
int fake_count(int d) { return count[d]; }
unsigned long fake_sum(int d) { return sum[d]; }
"""

CALL = r"""
import ctypes as C, sys
fake, lib = C.CDLL(sys.argv[1]), C.CDLL(sys.argv[2])
fake.fake_sum.restype = C.c_ulong
name, arg = sys.argv[3], sys.argv[4]
prepare = getattr(lib, "_ZN4tnbp%d%sE%s" % (len(name), name, arg))
for d in (0, 1, 1, 0):
    fake.fake_use(d)
    assert prepare(64) == 0
print(fake.fake_count(0), fake.fake_count(1), fake.fake_sum(0) == fake.fake_sum(1))
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    B.build()
    d = tmp_path_factory.mktemp("fake")
    src, so = d / "fake.c", d / "libfake.so"
    src.write_text(FAKE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    return str(so)


@pytest.mark.parametrize("name,calls", [
    ("simt_prepare", 8), ("site_sweep_prepare", 7), ("tc_prepare", 2), ("tc_stream_prepare", 7),
    ("normalise_prepare", 1), ("solve32_prepare", 1), ("basis_gmem_prepare", 3),
    ("refine_prepare", 5)])
def test_attributes_are_set_once_on_each_device(fake, name, calls):
    arg = "i" if name == "normalise_prepare" else "v"
    r = subprocess.run([sys.executable, "-c", CALL, fake, tn.LIB_PATH, name, arg],
                       env=dict(os.environ, LD_PRELOAD=fake), capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert r.stdout.split() == [str(calls), str(calls), "True"]
