"""The library works on after cudaDeviceReset: nothing it keeps beside handles (memory pool, pinned
status blocks, limits raised on kernels) is used in a later context.  Run in a child process,
since a reset also ends the context of everything else in the process."""

import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes, glob, sys, threading
import numpy as np
from paper_2411_06405_gb300 import _lib
from synth import erdos_renyi_gnm

lib = _lib.load()
found = sorted(glob.glob("/usr/local/cuda/lib64/libcudart.so.1[0-9]"))
if not found:
    sys.exit(77)
rt = ctypes.CDLL(found[0])
n = 300
s, d = erdos_renyi_gnm(n, 1200, 11)


def run(h):
    out = [np.zeros(s.size, np.int32) for _ in range(3)]
    m = ctypes.c_int64()
    p = lambda a: ctypes.c_void_p(a.ctypes.data)
    st = lib.htd_truss_decompose_host(n, p(s), p(d), s.size, h, *(p(a) for a in out), ctypes.byref(m), None, None)
    assert st == 0, lib.htd_last_error()
    return [a[:m.value] for a in out]


ref = {h: run(h) for h in (1, 2, 3, 4)}
for _ in range(2):
    assert rt.cudaSetDevice(0) == 0 and rt.cudaDeviceReset() == 0
    for h in (3, 2, 1, 4, 2):
        assert all(np.array_equal(a, b) for a, b in zip(run(h), ref[h])), h
    # a thread that has made no CUDA call before
    got = []
    th = threading.Thread(target=lambda: got.append(run(2)))
    th.start()
    th.join()
    assert all(np.array_equal(a, b) for a, b in zip(got[0], ref[2]))
print("same after reset")
"""


def test_works_after_device_reset():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2411_06405_gb300 import build

    build.build()
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=120)
    if r.returncode == 77:
        pytest.skip("no shared CUDA runtime to reset the device with")
    assert r.returncode == 0, r.stdout + r.stderr
    assert "same after reset" in r.stdout
