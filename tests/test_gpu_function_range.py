"""Gaussian and Lorentzian vertex values where (x - mu) / s leaves the range of a
double: the functions' limits (0), as the oracle gives them."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pwl():
    import paper_1510_02975_gb300 as m
    from paper_1510_02975_gb300 import _build
    _build.build()
    return m


@pytest.mark.parametrize("kind", ["gaussian", "lorentzian"])
@pytest.mark.parametrize("s,x", [(1e-10, 1e300), (-1e-10, 1e300), (1e-100, 1e250), (0.5, 1.7e308)])
def test_quotients_beyond_the_range(pwl, kind, s, x):
    f = {"kind": kind, "a": -x / 2, "b": x / 2, "p": [2.0, 0.0, s]}
    knots = np.array([-x / 2, -abs(s), 0.0, abs(s), x / 2])
    v = pwl.pwl_project(f, torch.tensor(knots, device="cuda"), "interp").cpu().numpy()
    ref = oracle.f_many(f, knots)
    assert ref[0] == 0.0 or kind == "lorentzian"
    assert np.all(np.isfinite(ref)) and np.all(np.abs(v - ref) <= 1e-15 * np.abs(ref).max()), (v, ref)
