"""The workspace of a single projection: 256 bytes, two doubles per interval and
four per knot, each array rounded up to 256 bytes -- what callers have sized
their buffers by -- is accepted and not overrun."""
import ctypes

import numpy as np
import pytest

import oracle
from pwl_testutil import VALUES_REL


def _size(n):
    return 256 + (16 * n + 255) // 256 * 256 + (32 * (n + 1) + 255) // 256 * 256


@pytest.fixture(scope="module")
def lib():
    from paper_1510_02975_gb300 import _build, _capi
    _build.build()
    return _capi.load()


@pytest.mark.parametrize("n", [1, 2, 7, 63, 64, 1024, 4095, 100001])
def test_size_asked_for(lib, n):
    assert lib.pwl_project_workspace_size(n) == _size(n)


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n", [1, 2, 63, 1024, 9000])  # the last one's solve works in the workspace
def test_nothing_is_written_past_it(lib, n, precision):
    torch = pytest.importorskip("torch")
    import paper_1510_02975_gb300 as pwl
    from paper_1510_02975_gb300 import _capi
    f = {"kind": "gaussian", "a": -4.0, "b": 4.0, "p": [1.0, 0.0, 1.0]}
    knots = pwl.pwl_design(f, n)
    values = torch.empty_like(knots)
    ws = torch.full((_size(n) + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    fn = _capi.make_func(f)
    st = lib.pwl_project(ctypes.byref(fn), knots.data_ptr(), n, 1, 8, {"fp64": 0, "fp32": 1}[precision],
                         values.data_ptr(), ws.data_ptr(), _size(n), torch.cuda.current_stream().cuda_stream)
    assert st == 0, lib.pwl_last_error()
    assert bool((ws[_size(n):] == 0xA5).all())
    if precision == "fp64":
        ref = oracle.values(f, knots.cpu().numpy(), "project")
        assert np.abs(values.cpu().numpy() - ref).max() <= VALUES_REL * np.abs(ref).max()
