"""The P_T paths a launch chooses between -- one thread or 16 lanes per
interval, partitioned solve with and without the recurrence over its blocks --
against the oracle (Eqs. 4-6), within the FP64 bound."""
import numpy as np
import pytest

import oracle
from pwl_testutil import VALUES_REL

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# block sizes of the partitioned solve from one row to 128, and their edges
SIZES = [1, 2, 3, 4, 31, 62, 63, 64, 65, 100, 999, 1599, 1600, 1663, 1700, 2047, 2500, 4095]


@pytest.fixture(scope="module")
def pwl():
    import paper_1510_02975_gb300 as m
    from paper_1510_02975_gb300 import _build
    _build.build()
    return m


def _check(pwl, funcs, n_int):
    b = pwl.Batch(funcs, n_int, m_per_interval=8)
    b.design()
    b.project("project")
    knots, values, off = b.knots().cpu().numpy(), b.values().cpu().numpy(), b.offsets()
    for i, f in enumerate(funcs):
        k, v = knots[off[i]:off[i + 1]], values[off[i]:off[i + 1]]
        ref = oracle.values(f, k, "project")
        assert np.abs(v - ref).max() <= VALUES_REL * np.abs(ref).max(), (f["kind"], n_int[i])


@pytest.mark.parametrize("copies", [1, 4])
def test_partitioned_solve_sizes(pwl, copies):
    # 4 copies: more intervals than the 16-lane quadrature serves
    kinds = [{"kind": "gaussian", "a": -4.0, "b": 4.0, "p": [1.0, 0.0, 0.7]},
             {"kind": "lorentzian", "a": -10.0, "b": 10.0, "p": [2.0, 0.5, 1.3]},
             {"kind": "bessel_j0", "a": 0.0, "b": 50.0, "p": [1.0, 4.0]},
             {"kind": "exp", "a": 0.0, "b": 10.0, "p": [1.0, 5.0]}]  # 22 decades
    n_int = SIZES * 4 * copies
    _check(pwl, [kinds[i // len(SIZES) % 4] for i in range(len(n_int))], n_int)


def test_gaussian_width_whose_reciprocal_is_not_normal(pwl):
    # s = 1e-300: 1/s^2 overflows, so the kernels divide
    f = {"kind": "gaussian", "a": -4e-300, "b": 4e-300, "p": [1.0, 0.0, 1e-300]}
    v = pwl.pwl_project(f, torch.tensor([-4e-300, -1e-300, 0.0, 2e-300, 4e-300], dtype=torch.float64, device="cuda"),
                        "interp").cpu().numpy()
    assert np.abs(v - np.exp(-0.5 * np.array([-4.0, -1.0, 0.0, 2.0, 4.0]) ** 2)).max() <= 1e-15
