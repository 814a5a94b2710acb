"""A push while another device is current is refused before anything is
launched (its kernels would run there, on this stream's memory).  On the CPU,
with the runtime's calls replaced by a counting stand-in."""
import os
import shutil
import subprocess
import sys
import textwrap

import pytest

import paper_1411_5373_gb300 as FD

STAND_IN = """
#include <stdlib.h>
#include <string.h>
int stand_in_device = 0, stand_in_launches = 0;
int cudaGetDevice(int *d) { *d = stand_in_device; return 0; }
int cudaSetDevice(int d) { return 0; }
int cudaMalloc(void **p, size_t n) { *p = aligned_alloc(256, (n + 255) / 256 * 256); return *p ? 0 : 2; }
int cudaFree(void *p) { free(p); return 0; }
int cudaMemcpy(void *d, const void *s, size_t n, int k) { memcpy(d, s, n); return 0; }
int cudaMemset(void *d, int v, size_t n) { memset(d, v, n); return 0; }
int cudaMemset2D(void *d, size_t p, int v, size_t w, size_t h) { return 0; }
int cudaGetLastError(void) { return 0; }
int cudaLaunchKernel(void) { ++stand_in_launches; return 0; }
int __cudaLaunchKernel(void) { ++stand_in_launches; return 0; }
int __cudaGetKernel(void **k, const void *f) { *k = (void *)f; return 0; }
"""

CALL = """
import ctypes
import sys
import paper_1411_5373_gb300 as FD
from paper_1411_5373_gb300 import _native as N
lib = FD.load()
fake = ctypes.CDLL(sys.argv[1])
device = ctypes.c_int.in_dll(fake, "stand_in_device")
launches = ctypes.c_int.in_dll(fake, "stand_in_launches")
for flags in (N.SCHED_PLAIN, N.SCHED_FUSED):
    s = ctypes.c_void_p()
    assert lib.fdmt_stream_create(1200.0, 1600.0, 16, 64, 20, N.F32_F32, flags, ctypes.byref(s)) == N.OK
    raw = ctypes.create_string_buffer(64 * 20 * 4 + 16)
    at = (ctypes.addressof(raw) + 15) // 16 * 16
    device.value = 1
    assert lib.fdmt_stream_push(s, at, at, None) == N.ERR_INVALID_ARG
    assert launches.value == 0, "launched on another device"
    device.value = 0
    lib.fdmt_stream_destroy(s)
print("refused")
"""


def test_push_on_another_device_launches_nothing(tmp_path, repo_root):
    cc = shutil.which("gcc")
    if cc is None or not os.path.exists(FD._native.LIB_PATH):
        pytest.skip("needs gcc and the built library")
    src, so = tmp_path / "stand_in.c", tmp_path / "stand_in.so"
    src.write_text(STAND_IN)
    subprocess.run([cc, "-shared", "-fPIC", "-w", "-o", str(so), str(src)], check=True)
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(CALL), str(so)], cwd=repo_root, capture_output=True,
                       text=True, env={**os.environ, "LD_PRELOAD": str(so)})
    assert r.returncode == 0 and r.stdout.split() == ["refused"], r.stderr
