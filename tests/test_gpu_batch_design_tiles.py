"""The FP32 design of a batch (2048-cell tiles) against the FP64 oracle at the
edges of tiles and vectors, and independent of what else is in the batch."""
import numpy as np
import pytest

import oracle
from pwl_testutil import fp32_design_bound

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

F_ALL = [{"kind": "gaussian", "a": -4.0, "b": 4.0, "p": [1.0, 0.0, 1.0]},
         {"kind": "lorentzian", "a": -10.0, "b": 10.0, "p": [1.0, 0.0, 1.0]},
         {"kind": "bessel_j0", "a": 0.0, "b": 50.0, "p": [1.0, 1.0]}]


@pytest.fixture(scope="module")
def pwl():
    import paper_1510_02975_gb300 as m
    from paper_1510_02975_gb300 import _build
    _build.build()
    return m


def _knots(pwl, funcs, n_int, mper):
    b = pwl.Batch(funcs, n_int, m_per_interval=mper)
    b.design("fp32")
    k, off = b.knots().cpu().numpy(), b.offsets()
    return [k[off[i]:off[i + 1]] for i in range(len(funcs))]


@pytest.mark.parametrize("mper", [16, 63])
def test_tile_edges(pwl, mper):
    # cell counts around multiples of 4 (a vector), 8 (a thread) and 2048 (a tile)
    n_int = [33, 65, 127, 128, 129, 255, 256, 257, 512, 641]
    funcs = [F_ALL[i % 3] for i in range(len(n_int))]
    for f, n, k in zip(funcs, n_int, _knots(pwl, funcs, n_int, mper)):
        ref = oracle.design(f, n, mper * n)
        assert np.all(np.abs(k - ref) <= fp32_design_bound(ref)), (f["kind"], n)


def test_independent_of_the_rest_of_the_batch(pwl):
    # the same function alone, first, last and among others: the same bits
    n_int = [1, 2, 3, 700, 5, 130, 1]
    funcs = [F_ALL[i % 3] for i in range(len(n_int))]
    together = _knots(pwl, funcs, n_int, 17)
    for f, n, k in zip(funcs, n_int, together):
        assert np.array_equal(k, _knots(pwl, [f], [n], 17)[0]), n


def test_linear_and_sampled_functions_among_analytic_ones(pwl):
    S = 4097
    x = np.linspace(-4.0, 4.0, S)
    smp = np.exp(-0.5 * x * x)
    line = {"kind": "poly", "a": -1.0, "b": 2.0, "p": [0.5, 2.0]}
    gpu = [F_ALL[0], line, {"kind": "sampled", "a": -4.0, "b": 4.0, "samples": torch.tensor(smp, device="cuda")}, F_ALL[2]]
    ref = [F_ALL[0], line, {"kind": "sampled", "a": -4.0, "b": 4.0, "samples": smp}, F_ALL[2]]
    n_int = [150, 150, 300, 40]
    for f, n, k in zip(ref, n_int, _knots(pwl, gpu, n_int, 32)):
        r = oracle.design(f, n, 32 * n)
        assert np.all(np.abs(k - r) <= fp32_design_bound(r)), (f["kind"], n)
