"""The FP64 design's tiled kernels (256-cell chunks, 2048-cell tiles) at the
edges of chunks and tiles, across runs of zero density that span tiles, and
as a batch: against the oracle (Eqs. 16-18)."""
import numpy as np
import pytest

import oracle
from pwl_testutil import DESIGN_REL

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GAUSS = {"kind": "gaussian", "a": -4.0, "b": 4.0, "p": [1.0, 0.0, 1.0]}
WIDE = {"kind": "gaussian", "a": -300.0, "b": 500.0, "p": [1.0, 0.0, 1.0]}  # f'' underflows to 0 past |x| ~ 38
CELLS = [1, 2, 255, 256, 257, 2047, 2048, 2049, 4095, 4097, 6145]


@pytest.fixture(scope="module")
def pwl():
    import paper_1510_02975_gb300 as m
    from paper_1510_02975_gb300 import _build
    _build.build()
    return m


@pytest.mark.parametrize("func", [GAUSS, WIDE], ids=["gaussian", "wide"])
@pytest.mark.parametrize("cells", CELLS)
def test_single_design_at_tile_edges(pwl, func, cells):
    for n in (1, 7, 300):
        got = pwl.pwl_design(func, n, cells).cpu().numpy()
        ref = oracle.design(func, n, cells)
        assert np.abs(got - ref).max() <= DESIGN_REL * (func["b"] - func["a"]), n


def test_batch_design_equals_single_design(pwl):
    # the same kernels, so the same bits: functions of every tile count, largest last and first
    n_int = [1, 3, 4, 31, 32, 33, 64, 65, 500, 2, 1000, 1]
    funcs = [GAUSS if i % 2 else WIDE for i in range(len(n_int))]
    b = pwl.Batch(funcs, n_int, m_per_interval=64)
    b.design()
    knots, off = b.knots(), b.offsets()
    for i, (f, n) in enumerate(zip(funcs, n_int)):
        assert torch.equal(knots[off[i]:off[i + 1]], pwl.pwl_design(f, n, 64 * n)), i


def test_knot_on_a_plateau_of_zero_density(pwl):
    # f'' is zero on the middle third (10923 of 32768 cells, five tiles): the
    # middle knot's target ties with the plateau's G, so it sits at one of the
    # plateau's ends (which one is rounding), never inside
    S, third = 3073, 1024
    j = np.arange(S)
    s = np.where(j < third, (third - j) ** 2.0, np.where(j > 2 * third, (j - 2 * third) ** 2.0, 0.0))
    f = {"kind": "sampled", "a": 0.0, "b": 3.0, "samples": torch.tensor(s, device="cuda")}
    for n in (2, 4):
        x = float(pwl.pwl_design(f, n, 32768)[n // 2])
        assert min(abs(x - 1.0), abs(x - 2.0)) <= 2.0 / third, x
