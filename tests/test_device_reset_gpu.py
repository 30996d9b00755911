"""What the library sets on a device (the shared-memory limits of its kernels) holds for the
context it was set in: after cudaDeviceReset, and so on a second device, the calls that
split or aggregate in shared memory work as they did before.  Runs in a process of its own
without PyTorch's CUDA state."""
from __future__ import annotations

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import ctypes
import numpy as np
from paper_2009_07914_gb300 import build
build.build()
from paper_2009_07914_gb300 import api

rt = ctypes.CDLL("libcudart.so.13")


def device(a):
    p = ctypes.c_void_p()
    assert rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(a.nbytes)) == 0
    assert rt.cudaMemcpy(p, ctypes.c_void_p(a.ctypes.data), ctypes.c_size_t(a.nbytes), 1) == 0
    return p.value


def host(p, n, dtype):
    a = np.empty(n, dtype)
    assert rt.cudaMemcpy(ctypes.c_void_p(a.ctypes.data), ctypes.c_void_p(p), ctypes.c_size_t(a.nbytes), 2) == 0
    return a


def run():
    n, big = 400_000, (1 << 24) + 5
    keys = (np.arange(1, big + 1, dtype=np.uint64) * 0x9E3779B1).astype(np.uint32)
    k, out, found = device(keys), device(np.zeros(n, np.uint32)), device(np.zeros(n, np.uint8))
    for insert in (api.wc_insert, api.wc_insert_noalloc):  # split by region
        t = api.wc_table_create(0, 4, 4, 9_000_000, 8, device=0)
        insert(t, k, k, n, stream=0)
        api.wc_retrieve(t, k, out, found, n, stream=0)
        assert (host(out, n, np.uint32) == keys[:n]).all() and host(found, n, np.uint8).all()
        api.wc_table_destroy(t)
    t = api.wc_table_create(4, 4, 4, 1_000_000, 8, device=0)  # counting
    api.wc_insert(t, k, None, n, stream=0)
    api.wc_insert(t, k, None, 1000, stream=0)
    api.wc_retrieve(t, k, out, found, n, stream=0)
    assert (host(out, n, np.uint32) == np.where(np.arange(n) < 1000, 2, 1)).all()
    api.wc_table_destroy(t)
    t = api.wc_table_create(1, 4, 4, 1_000_000, 4, 3 * n, device=0)  # bucket multi-value
    api.wc_insert(t, k, k, n, stream=0)
    assert api.wc_size(t, stream=0) == n
    api.wc_table_destroy(t)
    t = api.wc_table_create(5, 4, 0, 10 << 20, 7, device=0)  # Bloom filter, filled by region
    api.wc_insert(t, k, None, big, stream=0)
    api.wc_contains(t, k, found, n, stream=0)
    assert host(found, n, np.uint8).all() and api.wc_size(t, stream=0) == big
    api.wc_table_destroy(t)


for _ in range(2):
    run()
    assert rt.cudaDeviceReset() == 0
print("done")
"""


def test_calls_work_again_after_a_device_reset():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=root, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and r.stdout.strip() == "done", r.stdout + r.stderr
