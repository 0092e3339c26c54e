"""A destroyed table's memory is reused in the context it was allocated in and in
no other: tables built, used and destroyed in a second context of the device
between two of the first.  In a process of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import ctypes, numpy as np, torch
import paper_1510_02975_gb300 as pwl
from paper_1510_02975_gb300 import _capi
lib, cu = _capi.load(), ctypes.CDLL("libcuda.so.1")
N, M = 63, 4096
k = np.linspace(-4, 4, N + 1); v = np.sin(k)
x = np.linspace(-5, 5, M).astype(np.float32)

def first():
    t = pwl.Table(torch.tensor(k, device="cuda"), torch.tensor(v, device="cuda"))
    y = t(torch.tensor(x, device="cuda")).cpu().numpy()
    t.close()
    return y

def ok(e):
    assert e == 0, e

def second():
    def up(a):
        d = ctypes.c_uint64()
        ok(cu.cuMemAlloc_v2(ctypes.byref(d), ctypes.c_size_t(a.nbytes)))
        ok(cu.cuMemcpyHtoD_v2(d, ctypes.c_void_p(a.ctypes.data), ctypes.c_size_t(a.nbytes)))
        return d
    dk, dv, dx, dy = up(k), up(v), up(x), up(np.zeros_like(x))
    ys = []
    for _ in range(3):
        h = ctypes.c_void_p()
        ok(lib.pwl_table_build(dk.value, dv.value, N, 0, 0, ctypes.byref(h), None))
        ok(lib.pwl_eval(h, dx.value, dy.value, M, 0, None))
        y = np.empty_like(x)
        ok(cu.cuMemcpyDtoH_v2(ctypes.c_void_p(y.ctypes.data), dy, ctypes.c_size_t(y.nbytes)))
        ok(lib.pwl_table_destroy(h))
        ys.append(y)
    for d in (dk, dv, dx, dy):
        ok(cu.cuMemFree_v2(d))
    return ys

want = first()
ctx, old = ctypes.c_void_p(), ctypes.c_void_p()
ok(cu.cuCtxCreate_v2(ctypes.byref(ctx), 0, 0))
ys = second()
ok(cu.cuCtxPopCurrent_v2(ctypes.byref(old)))
ys += [first(), first()]
ok(cu.cuCtxDestroy_v2(ctx))
ys.append(first())
assert all(np.array_equal(y, want) for y in ys)
print("same")
"""


def test_second_context():
    pytest.importorskip("torch")
    from paper_1510_02975_gb300 import _build
    _build.build()
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same" in r.stdout, r.stderr[-2000:]
