"""Builds in a second context of a device, and in a primary context made anew
after a reset: what the library keeps between builds belongs to the context that
it was made in.  Runs in a process of its own, which has no other CUDA user."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes as C
import glob
import numpy as np
from paper_2411_12365_gb300 import burr
from paper_2411_12365_gb300 import inputs as I

cu = C.CDLL("libcuda.so.1")


def context_id():
    c, i = C.c_void_p(), C.c_ulonglong(0)
    cu.cuCtxGetCurrent(C.byref(c))
    return i.value if cu.cuCtxGetId(c, C.byref(i)) == 0 else 0


n = 20_011
k = I.keys_np(n, seed=5)
v = I.values_np(k, 8)
big = np.concatenate([k] * 420)   # a host batch past the size that one stream takes


def check():
    h = burr.build(k, v, 8)
    assert np.array_equal(h.query(k), v)
    assert np.array_equal(h.query(big)[-n:], v)
    ex = h.export()
    h.free()
    return ex


want = check()
assert check() == want
first = context_id()
assert first
second = C.c_void_p()
assert cu.cuCtxCreate_v2(C.byref(second), 0, 0) == 0
assert context_id() not in (0, first)
assert check() == want and check() == want
assert cu.cuCtxPopCurrent_v2(C.byref(C.c_void_p())) == 0
assert context_id() == first
assert check() == want
assert cu.cuCtxDestroy_v2(second) == 0
assert check() == want
for _ in range(12):   # more contexts than sets are kept
    assert cu.cuCtxCreate_v2(C.byref(second), 0, 0) == 0
    assert check() == want
    assert cu.cuCtxDestroy_v2(second) == 0
assert check() == want
print("contexts ok", flush=True)

runtimes = glob.glob("/usr/local/cuda/lib64/libcudart.so.*")
if runtimes:
    rt = C.CDLL(sorted(runtimes)[0])
    assert rt.cudaSetDevice(0) == 0 and rt.cudaDeviceReset() == 0
    assert rt.cudaSetDevice(0) == 0 and rt.cudaFree(None) == 0
    assert context_id() not in (0, first)   # what the library tells contexts apart by
    assert check() == want and check() == want
    print("reset ok", flush=True)
"""


def test_second_context_and_reset():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "contexts ok" in r.stdout
