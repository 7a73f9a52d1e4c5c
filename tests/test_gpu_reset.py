"""A device reset between two sets: every handle of the first context is
destroyed before it, and a set built after it works.  In a process of its own,
which the reset ends nothing for but its own context.  Memory through the CUDA
runtime alone: no other library's context is on the device then."""
import subprocess
import sys

import pytest

from paper_2305_05055_gb300 import build

pytestmark = pytest.mark.gpu

PROGRAM = r"""
import ctypes as C, sys
V, U = C.c_void_p, C.c_uint64
rt, L = C.CDLL(sys.argv[1]), C.CDLL(sys.argv[2])

def go(n, handles):
    key, s = V(), V()
    a = (U * n)(*[i * 977 + 5 for i in range(n)])
    assert rt.cudaMalloc(C.byref(key), U(8 * n)) == 0 and rt.cudaMalloc(C.byref(s), U(16)) == 0
    assert rt.cudaMemcpy(key, a, U(8 * n), 1) == 0
    hs = []
    for _ in range(handles):
        h, size = V(), U()
        assert L.cpma_create(C.byref(h), None, key, U(n), V(0)) == 0
        assert L.cpma_size(h, C.byref(size)) == 0 and size.value == n
        assert L.cpma_sum(h, s, V(s.value + 8), V(0)) == 0
        o = (U * 2)()
        assert rt.cudaMemcpy(o, s, U(16), 2) == 0 and o[0] == sum(a) and o[1] == n
        hs.append(h)
    for h in hs:
        assert L.cpma_destroy(h) == 0

go(3000, 3)
for _ in range(2):
    assert rt.cudaDeviceReset() == 0
    go(2000, 70)   # more handles at once than the library keeps status blocks for
print("done")
"""


def test_a_set_after_a_device_reset():
    rt = "/usr/local/cuda/lib64/libcudart.so"
    try:
        import ctypes
        ctypes.CDLL(rt)
    except OSError:
        pytest.skip("no CUDA runtime library to reset the device with")
    r = subprocess.run([sys.executable, "-c", PROGRAM, rt, build.LIB], capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "done", r.stdout + r.stderr
