"""Vertex values near the ends of the number ranges, as the oracle gives them:
Gaussians and Lorentzians where (x - mu) / s leaves the range of a double (their
limit, 0), and FP32 integrands between knots whose sum leaves FP32's."""
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


@pytest.mark.parametrize("a,b,mu,s", [(2e38, 3e38, 2.4e38, 2e37), (-3e38, -2e38, -2.4e38, 2e37), (-3e38, 3e38, 0.0, 2e38)])
def test_fp32_integrand_between_large_knots(pwl, a, b, mu, s):
    f = {"kind": "gaussian", "a": a, "b": b, "p": [1.0, mu, s]}
    for n in (1, 2, 40):
        knots = np.linspace(a, b, n + 1)
        v = pwl.pwl_project(f, torch.tensor(knots, device="cuda"), "project", precision="fp32").cpu().numpy()
        ref = oracle.values(f, knots, "project")
        # f at FP32-rounded points: |t f'(t)| 2^-24 <= |t| / s 2^-24 each, 2.5 of that after the solve
        assert np.all(np.abs(v - ref) <= 2.5 * (max(abs(a), abs(b)) / s * 2.0 ** -24 + 2.0 ** -22)), n
