"""The batch index built in shared memory, and in global memory where a
function is too large for it: evaluations against the oracle, with cells
that hold no knot, one and several."""
import numpy as np
import pytest

import oracle
from pwl_testutil import EVAL_REL

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pwl():
    import paper_1510_02975_gb300 as m
    from paper_1510_02975_gb300 import _build
    _build.build()
    return m


@pytest.mark.parametrize("cells_per_knot", [1, 3, 12])
@pytest.mark.parametrize("n_int", [[1, 2, 1023, 1024, 1025, 4095], [14000, 7], [20000, 3, 500]],
                         ids=["staged", "one_cta", "global"])
def test_index_records(pwl, n_int, cells_per_knot):
    kinds = [{"kind": "gaussian", "a": -4.0, "b": 4.0, "p": [1.0, 0.0, 1.0]},
             {"kind": "lorentzian", "a": -10.0, "b": 10.0, "p": [1.0, 0.0, 1.0]}]
    funcs = [kinds[i % 2] for i in range(len(n_int))]
    b = pwl.Batch(funcs, n_int, m_per_interval=4, cells_per_knot=cells_per_knot)
    b.design()
    b.project("interp")
    b.build()
    xk, vk, off = b.knots_fp32().cpu().numpy(), b.values_fp32().cpu().numpy(), b.offsets()
    rng = np.random.default_rng(1)
    xs = [np.concatenate([rng.uniform(f["a"] - 0.5, f["b"] + 0.5, 20000), xk[off[i]:off[i + 1]]]).astype(np.float32)
          for i, f in enumerate(funcs)]
    qo = np.concatenate([[0], np.cumsum([x.size for x in xs])])
    b.plan(qo)
    y = b.eval(torch.tensor(np.concatenate(xs), device="cuda")).cpu().numpy().astype(np.float64)
    b.check()
    for i in range(len(funcs)):
        k, v = xk[off[i]:off[i + 1]].astype(np.float64), vk[off[i]:off[i + 1]].astype(np.float64)
        ref = oracle.evaluate(k, v, xs[i].astype(np.float64))
        assert np.abs(y[qo[i]:qo[i + 1]] - ref).max() <= EVAL_REL * np.abs(v).max(), n_int[i]
