"""The batch index where one interval spans most of a function's cells (a long
part without curvature): evaluations against the oracle, and a build that takes
no longer for it than a few builds of evenly spread knots."""
import numpy as np
import pytest

import oracle
from pwl_testutil import EVAL_REL

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SMOOTH = {"kind": "gaussian", "a": -4.0, "b": 4.0, "p": [1.0, 0.0, 1.0]}
# knots in [-4, ~6] only: the density underflows further out
GAP = {"kind": "gaussian", "a": -4.0, "b": 400.0, "p": [1.0, 0.0, 1.0]}
GAP_LEFT = {"kind": "gaussian", "a": -400.0, "b": 4.0, "p": [1.0, 0.0, 1.0]}


@pytest.fixture(scope="module")
def pwl():
    import paper_1510_02975_gb300 as m
    from paper_1510_02975_gb300 import _build
    _build.build()
    return m


def _built(pwl, funcs, n_int, cells):
    b = pwl.Batch(funcs, n_int, m_per_interval=64, cells_per_knot=cells)
    b.design()
    b.project("interp")
    b.build()
    b.check()
    return b


@pytest.mark.parametrize("n_int,cells", [([1, 2, 31, 32, 33, 1023, 1024, 4095], 12), ([300] * 8, 64), ([20000, 40], 20)])
def test_values_in_and_beside_the_gap(pwl, n_int, cells):
    funcs = [(GAP, GAP_LEFT)[i % 2] for i in range(len(n_int))]
    b = _built(pwl, funcs, n_int, cells)
    xk, vk, off = b.knots_fp32().cpu().numpy(), b.values_fp32().cpu().numpy(), b.offsets()
    rng = np.random.default_rng(1)
    xs = [np.concatenate([rng.uniform(f["a"], f["b"], 20000), rng.uniform(-6, 6, 20000), xk[off[i]:off[i + 1]]])
          .astype(np.float32) for i, f in enumerate(funcs)]
    qo = np.concatenate([[0], np.cumsum([x.size for x in xs])])
    b.plan(qo)
    y = b.eval(torch.tensor(np.concatenate(xs), device="cuda")).cpu().numpy().astype(np.float64)
    for i in range(len(funcs)):
        k, v = xk[off[i]:off[i + 1]].astype(np.float64), vk[off[i]:off[i + 1]].astype(np.float64)
        ref = oracle.evaluate(k, v, xs[i].astype(np.float64))
        assert np.abs(y[qo[i]:qo[i + 1]] - ref).max() <= EVAL_REL * np.abs(v).max(), n_int[i]


@pytest.mark.parametrize("functions,n,cells", [(300, 4095, 4), (40, 4095, 64), (1, 20000, 64)])
def test_build_time(pwl, functions, n, cells):
    def us(f):
        b = _built(pwl, [f] * functions, [n] * functions, cells)
        times = []
        for _ in range(10):
            a, e = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            b.build()
            e.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(e) * 1e3)
        b.close()
        return sorted(times)[4]

    smooth, gap = us(SMOOTH), us(GAP)
    assert gap <= 3.0 * smooth, (gap, smooth)
