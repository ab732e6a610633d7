"""Both compaction entry points after a device reset, in a process of its own (the
reset ends that process's context only): nothing of the context before is used."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes, glob, os, sys
import numpy as np
from paper_2308_01241_gb300 import dtb

rt = ctypes.CDLL(sys.argv[1])
rt.cudaMalloc.argtypes = [ctypes.c_void_p, ctypes.c_size_t]
rt.cudaMemcpy.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int]


def ok(r):
    assert r == 0, f"CUDA error {r}"


n = 200_003
for turn in range(3):
    fired = np.random.default_rng(turn).random(n) < 0.01
    pad = np.zeros(-(-n // 1024) * 1024, bool)
    pad[:n] = fired
    bits = np.packbits(pad, bitorder="little")
    want = np.flatnonzero(fired)
    d = [ctypes.c_void_p() for _ in range(3)]
    for p, size in zip(d, (bits.nbytes, 4 * n, 4)):
        ok(rt.cudaMalloc(ctypes.byref(p), size))
    ok(rt.cudaMemcpy(d[0], bits.ctypes.data, bits.nbytes, 1))
    for call in (dtb._lib.dtb_spike_compact_noalloc, dtb._lib.dtb_spike_compact, dtb._lib.dtb_spike_compact):
        dtb._check(call(d[0], n, d[1], d[2], None), "compaction")
        ids, cnt = np.full(n, -1, np.int32), np.zeros(1, np.int32)
        ok(rt.cudaMemcpy(ids.ctypes.data, d[1], ids.nbytes, 2))
        ok(rt.cudaMemcpy(cnt.ctypes.data, d[2], 4, 2))
        assert cnt[0] == want.size and (ids[: want.size] == want).all()
    ok(rt.cudaDeviceReset())
print("child ok")
"""


def test_compaction_after_a_device_reset():
    names = ("libcudart.so.13", "libcudart.so")
    dirs = [os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "lib64")]
    paths = [os.path.join(d, n) for d in dirs for n in names if os.path.exists(os.path.join(d, n))]
    if not paths:
        pytest.skip("no CUDA runtime library to reset the device with")
    r = subprocess.run([sys.executable, "-c", CHILD, paths[0]], cwd=ROOT, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "child ok" in r.stdout, r.stderr[-2000:]
