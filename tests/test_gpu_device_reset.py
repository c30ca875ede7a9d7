"""A program that resets its device between two phases (which ends its own
context only): queries on a new graph work as on the first one."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
import ctypes, sys
import numpy as np
import oracle as O
from paper_2506_19349_gb300 import binding, graphgen as G

L = binding.load_library()
C = ctypes.CDLL("libcudart.so.13")
wl = G.urand(12, 15, seed=5, nsources=2)
og = O.Graph(wl.n, wl.src, wl.dst, wl.w)
src, dst, w = (np.ascontiguousarray(x, np.uint32) for x in (wl.src, wl.dst, wl.w))

def phase(close):
    handles = []
    out = ctypes.c_void_p()
    assert C.cudaHostAlloc(ctypes.byref(out), ctypes.c_size_t(4 * wl.n), 2) == 0  # (mapped)
    for _ in range(3):
        h = ctypes.c_void_p()
        rc = L.eic_graph_create(src.ctypes.data, dst.ctypes.data, w.ctypes.data, src.size, wl.n, 0, None, ctypes.byref(h))
        assert rc == 0, rc
        handles.append(h)
    for _ in range(2):
        for h in handles:
            for s in wl.sources:
                rc = L.eic_sssp(h, int(s), out, None, None, None, None)
                assert rc == 0, rc
                got = np.ctypeslib.as_array(ctypes.cast(out, ctypes.POINTER(ctypes.c_uint32)), (wl.n,))
                assert np.array_equal(got, og.dijkstra(int(s))[0])
    if close:
        for h in handles:
            assert L.eic_graph_destroy(h) == 0

for close in (True, False, True):
    phase(close)
    assert C.cudaDeviceReset() == 0
phase(True)
print("reset ok")
"""


def test_queries_after_a_device_reset():
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "reset ok" in r.stdout, r.stdout + r.stderr
