"""Designs whose knots crowd into few density cells (few cells per knot, narrow
peaks) or spread evenly (no curvature), with tiles shared by several CTAs and
densities by whole tiles: parity with the oracle, every knot written once, and
a time that does not hang on where the knots lie."""
import numpy as np
import pytest

import oracle
from pwl_testutil import DESIGN_REL

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pwl():
    import paper_1510_02975_gb300 as m
    from paper_1510_02975_gb300 import _build
    _build.build()
    return m


def _peak(s):
    return {"kind": "gaussian", "a": -1.0, "b": 1.0, "p": [1.0, 0.1, s]}


LINEAR = {"kind": "poly", "a": -1.0, "b": 3.0, "p": [2.0, 0.5, 0, 0, 0, 0, 0, 0]}


@pytest.mark.parametrize("f", [_peak(0.3), _peak(1e-3), LINEAR], ids=["wide", "peak", "linear"])
@pytest.mark.parametrize("n,m", [(513, 2048), (1025, 300), (4096, 4096), (20000, 2049), (100000, 5000), (3000, 1 << 20)])
def test_knots(pwl, f, n, m):
    k = torch.full((n + 1,), float("nan"), dtype=torch.float64, device="cuda")
    pwl.pwl_design(f, n, m, knots=k)
    k = k.cpu().numpy()
    ref = oracle.design(f, n, m)
    # within the FP64 bound; where a cell holds many knots, up to its share of G's rounding
    assert np.all(np.abs(k - ref) <= DESIGN_REL * (f["b"] - f["a"])), np.abs(k - ref).max()
    assert np.all(np.diff(k) >= 0)


def test_fp32_densities_by_tiles(pwl):
    # more tiles than eight per SM: FP32 densities eight cells per thread
    f, n = _peak(0.2), 2000
    m = 1217 * 2048 - 777
    k = pwl.pwl_design(f, n, m, precision="fp32").cpu().numpy()
    ref = oracle.design(f, n, m)
    h = np.diff(ref)
    assert np.all(np.abs(k - ref) <= 2e-3 * np.minimum(np.r_[h[0], h], np.r_[h, h[-1]]))


def _us(call):
    call()
    times = []
    for _ in range(7):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        call()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b) * 1e3)
    return sorted(times)[3]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_time_of_few_cells_per_knot(pwl, precision):
    n = (1 << 20) - 1
    few = _us(lambda: pwl.pwl_design(_peak(0.3), n, 2048, precision=precision))
    many = _us(lambda: pwl.pwl_design(_peak(0.3), n, 64 * n, precision=precision))
    assert few <= 0.5 * many, (few, many)


@pytest.mark.parametrize("n", [100000, (1 << 20) - 1])
def test_time_of_a_peak(pwl, n):
    wide, peak = (_us(lambda: pwl.pwl_design(_peak(s), n)) for s in (0.3, 1e-4))
    assert peak <= 1.5 * wide, (peak, wide)


def test_time_of_fp32_densities(pwl):
    # an FP32 cell takes a fraction of an FP64 one: 16 M cells, few knots
    fp64, fp32 = (_us(lambda: pwl.pwl_design(_peak(0.3), 4096, 1 << 24, precision=q)) for q in ("fp64", "fp32"))
    assert fp32 <= 0.32 * fp64, (fp32, fp64)
