"""The shared-memory opt-in of the any-size kernels belongs to a device.  On the
CPU, over a stand-in for the CUDA runtime calls of mf_residual_noalloc that
keeps the attribute per (device, kernel) and refuses a launch above 48 KB
without it, as a device does: the call works on every device it is made on,
on one that has lost its attributes, and after a call whose opt-in failed."""
import os
import subprocess
import sys

import pytest

from paper_1901_06531_gb300 import build

FAKE = r"""
#include <stddef.h>
#include <string.h>
typedef struct { unsigned x, y, z; } dim3;
static int dev, fail_next, launches, last, n;
static struct { int dev; const void* f; int bytes; } set[256];
void fake_device(int d) { dev = d; }
void fake_reset(void) { for (int i = 0; i < n; ++i) if (set[i].dev == dev) set[i].bytes = 0; }
void fake_fail_next(void) { fail_next = 1; }
int fake_launches(void) { return launches; }
int cudaGetDevice(int* d) { *d = dev; return 0; }
int cudaStreamGetDevice(void* s, int* d) { *d = dev; return 0; }
int cudaGetSymbolAddress(void** p, const void* s) { *p = (void*)(size_t)4096; return 0; }
int cudaMemcpyAsync(void* d, const void* s, size_t b, int k, void* st) { return 0; }
int cudaMemsetAsync(void* d, int v, size_t b, void* st) { return 0; }
int cudaStreamSynchronize(void* st) { return 0; }
int cudaGetLastError(void) { const int e = last; last = 0; return e; }
int cudaFuncGetAttributes(void* a, const void* f) { memset(a, 0, 64); return 1; }   /* unknown: the caller's default */
int cudaFuncSetAttribute(const void* f, int attr, int v) {
  if (attr != 8) return 1;   /* cudaFuncAttributeMaxDynamicSharedMemorySize */
  if (fail_next) { fail_next = 0; return 2; }
  for (int i = 0; i < n; ++i) if (set[i].dev == dev && set[i].f == f) { set[i].bytes = v; return 0; }
  set[n].dev = dev; set[n].f = f; set[n++].bytes = v;
  return 0;
}
/* what a <<<>>> launch calls (crt/device_functions.h) */
int __cudaGetKernel(const void** k, const void* f) { *k = f; return 0; }
int __cudaLaunchKernel(const void* f, dim3 g, dim3 b, void** args, size_t smem, void* st) {
  size_t most = 48 * 1024 - 1024;   /* the kernels' static part */
  for (int i = 0; i < n; ++i) if (set[i].dev == dev && set[i].f == f && (size_t)set[i].bytes > most) most = set[i].bytes;
  ++launches;
  return last = smem > most ? 1 : 0;
}
"""

CHILD = r"""
import ctypes, sys
import numpy as np
mf, fake = ctypes.CDLL(sys.argv[1]), ctypes.CDLL(sys.argv[2])
vp = ctypes.c_void_p
mf.mf_residual_noalloc.argtypes = [ctypes.c_int] * 3 + [vp] * 6
mask, pbar = np.zeros(9, np.uint8), np.zeros(9)
def call(nx, ny, nz):
    k = fake.fake_launches()
    st = mf.mf_residual_noalloc(nx, ny, nz, vp(1 << 20), mask.ctypes.data, pbar.ctypes.data, vp(1 << 30), None, None)
    return st, fake.fake_launches() - k
large = [(128, 64, 4), (96, 96, 16), (16, 16, 256), (128, 192, 2)]   # planes, a z-pass and the largest plane above 48 KB
fake.fake_fail_next()
assert call(128, 64, 4)[0] == 5                      # MF_CUDA_ERROR, not kept
for device in (0, 1, 0, 2):
    fake.fake_device(device)
    for shape in large + [(16, 16, 16), (72, 72, 8)]:
        r = call(*shape); assert r == (0, 3), (device, shape, r)
fake.fake_device(1)
fake.fake_reset()
for shape in large:
    r = call(*shape); assert r == (0, 3), ("after a reset", shape, r)
print("ok")
"""


def test_opt_in_on_every_device(tmp_path):
    src, so = tmp_path / "fake.c", tmp_path / "fake.so"
    src.write_text(FAKE)
    try:
        subprocess.run(["gcc", "-w", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    except FileNotFoundError:
        pytest.skip("no C compiler")
    res = subprocess.run([sys.executable, "-c", CHILD, build.build(), str(so)], capture_output=True, text=True,
                         timeout=120, env=dict(os.environ, LD_PRELOAD=str(so)))
    assert res.returncode == 0 and "ok" in res.stdout, res.stderr[-2000:]
