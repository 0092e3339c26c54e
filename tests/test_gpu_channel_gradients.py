"""Channel-wise table gradients relative to their own terms: every knot's sum is
held to GRAD_REL of the absolute sum of what was added to it, whatever the
channel's other gradients are, in tiles of every shape (16 and 8 channels);
sums that fill the integer words; gx written over gy."""
import numpy as np
import pytest

import oracle
from pwl_testutil import EVAL_REL, GRAD_REL

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# (channels, intervals, k_cells): 16- and 8-channel tiles in the backward, each in the
# part of shared memory that leaves the L1 room and in all of it
WIDTHS = [(20, 40, 0), (20, 330, 0), (20, 40, 1700), (10, 640, 0)]


@pytest.fixture(scope="module")
def pwl():
    import paper_1510_02975_gb300 as m
    from paper_1510_02975_gb300 import _build
    _build.build()
    return m


def _tables(C, N, seed=0):
    rng = np.random.default_rng(seed)
    knots = np.tile(np.linspace(-2.0, 3.0, N + 1), (C, 1))
    knots[:, 1:-1] += rng.uniform(-0.4, 0.4, (C, N - 1)) * (5.0 / N)
    return knots.astype(np.float32), rng.normal(size=(C, N + 1)).astype(np.float32)


def _data(case, C, N, R, knots):
    rng = np.random.default_rng(3)
    x = rng.uniform(-2.2, 3.2, (R, C)).astype(np.float32)
    g = rng.normal(size=(R, C))
    j = N // 2
    if case.startswith("bin"):  # one interval's gradients 2^-k of the channel's
        lo, hi = knots[:, j - 1], knots[:, j + 1]
        g = np.where((x >= lo) & (x < hi), g * 2.0 ** -int(case[3:]), g)
    elif case == "decades":  # |gy| a function of x, over 12 decades
        g *= 10.0 ** (12 * (np.clip(x, -2, 3) + 2) / 5 - 12)
    elif case == "sparse_channels":  # 1% nonzero, each channel its own magnitude
        g *= (rng.random((R, C)) < 0.01) * 10.0 ** -(np.arange(C) % 13)
    elif case == "lognormal":
        g *= np.exp(2 * rng.normal(size=(R, C)))
    elif case == "outliers":  # a few elements far beyond what the samples suggest
        g[777::4999] *= 1e9
        g[1234] *= 1e33
    elif case == "beside_a_knot":  # no point near knot j: both intervals' within 2^-16 of their far ends
        l, m, r = knots[:, j - 1], knots[:, j], knots[:, j + 1]
        t = np.float32(2.0 ** -16) * rng.random((R, C)).astype(np.float32)
        x = np.where((x > l) & (x < m), l + (m - l) * t, np.where((x >= m) & (x < r), r - (r - m) * t, x))
    return x, g.astype(np.float32)


def _grads(pwl, knots, values, x, gy, k_cells=0, out=None):
    kt, vt, xt, gt = (torch.tensor(a, device="cuda") for a in (knots, values, x, gy))
    gv, gk = torch.zeros_like(vt), torch.zeros_like(kt)
    gx = pwl.pwl_channels_backward(kt, vt, xt, gt, gt if out == "gy" else None, gv, gk, k_cells=k_cells)
    return gx.cpu().numpy(), gv.cpu().numpy(), gk.cpu().numpy()


def _check(knots, values, x, gy, gv, gk, channels):
    for c in channels:
        _, rv, rk, av, ak = oracle.evaluate_grad(knots[c].astype(np.float64), values[c].astype(np.float64),
                                                 x[:, c].astype(np.float64), gy[:, c].astype(np.float64))
        assert np.all(np.abs(gv[c] - rv) <= GRAD_REL * av), (c, np.max(np.abs(gv[c] - rv) / np.maximum(av, 1e-300)))
        assert np.all(np.abs(gk[c] - rk) <= GRAD_REL * ak), (c, np.max(np.abs(gk[c] - rk) / np.maximum(ak, 1e-300)))


@pytest.mark.parametrize("C,N,k_cells", WIDTHS, ids=["16", "16_all", "8", "8_all"])
@pytest.mark.parametrize("case", ["normal", "bin16", "bin20", "bin26", "bin31", "decades", "sparse_channels", "lognormal",
                                  "outliers", "beside_a_knot"])
def test_every_knot_relative_to_its_own_terms(pwl, case, C, N, k_cells):
    knots, values = _tables(C, N)
    x, gy = _data(case, C, N, 20000, knots)
    _, gv, gk = _grads(pwl, knots, values, x, gy, k_cells)
    _check(knots, values, x, gy, gv, gk, range(C))


@pytest.mark.parametrize("N", [387, 388, 517, 518, 602, 603, 1036, 1037, 1206, 1207, 1790])
def test_forward_shapes(pwl, N):
    # the edges of the forward's tile shapes, one cell per knot at each
    C, R = 21, 700
    knots, values = _tables(C, N)
    x = _data("normal", C, N, R, knots)[0]
    x[:3] = knots[:, [0, N // 2, N]].T
    kt, vt, xt = (torch.tensor(a, device="cuda") for a in (knots, values, x))
    y = pwl.pwl_channels_forward(kt, vt, xt).cpu().numpy().astype(np.float64)
    for c in range(C):
        v = values[c].astype(np.float64)
        ref = oracle.evaluate(knots[c].astype(np.float64), v, x[:, c].astype(np.float64))
        assert np.abs(y[:, c] - ref).max() <= EVAL_REL * np.abs(v).max(), c


@pytest.mark.parametrize("N", [1, 5])
def test_sums_that_fill_the_words(pwl, N):
    # a CTA takes all rows of a tile; gradients of one size, the largest of its
    # binade, in one interval: the words grow as fast as samples let them
    C, R = 2432, 30001
    knots, values = _tables(C, N)
    x = np.repeat((0.25 * knots[:, :1] + 0.75 * knots[:, 1:2]).T.astype(np.float32), R, axis=0)
    gy = np.full((R, C), 1.9999999, dtype=np.float32)
    gy[-1] = 7.5  # beyond the samples, inside the range
    _, gv, gk = _grads(pwl, knots, values, x, gy)
    _check(knots, values, x, gy, gv, gk, [0, 1, 15, 16, 1000, 2431])


def test_gx_over_gy(pwl):
    C, N, R = 200, 30, 40000
    knots, values = _tables(C, N)
    values *= 1e7  # gx far from gy in size
    x, gy = _data("normal", C, N, R, knots)
    ref = _grads(pwl, knots, values, x, gy)
    gx, gv, gk = _grads(pwl, knots, values, x, gy, out="gy")
    assert np.array_equal(gx, ref[0])
    _check(knots, values, x, gy, gv, gk, range(0, C, 7))


@pytest.mark.parametrize("case", ["lognormal", "first_rows_zero", "sparse", "very_sparse", "small_bin", "outliers",
                                  "outside"])
def test_time_does_not_hang_on_the_gradients(pwl, case):
    # events around the backward of [65536, 1024] x 257 knots: other distributions of gy, and a
    # third of the points outside the domain, within half as much again as N(0, 1) gradients
    C, N, R = 1024, 256, 65536
    knots, values = (torch.tensor(a, device="cuda") for a in _tables(C, N))
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn(R, C, generator=g, device="cuda")
    gy = torch.randn(R, C, generator=g, device="cuda")
    gx, gv, gk = torch.empty_like(x), torch.zeros_like(values), torch.zeros_like(knots)

    def us(x, gy):
        times = []
        for _ in range(8):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            pwl.pwl_channels_backward(knots, values, x, gy, gx, gv, gk)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) * 1e3)
        return sorted(times)[3]

    x.clamp_(-1.99, 2.99)
    base = us(x, gy)
    if case == "lognormal":
        gy *= torch.exp(2 * torch.randn(R, C, generator=g, device="cuda"))
    elif case == "first_rows_zero":
        gy.view(-1, 1024, C)[:, 0] = 0
    elif case in ("sparse", "very_sparse"):
        gy *= torch.rand(R, C, generator=g, device="cuda") < (0.01 if case == "sparse" else 0.001)
    elif case == "small_bin":
        gy[(x > 0.5) & (x < 0.6)] *= 2.0 ** -26
    elif case == "outliers":
        gy[torch.rand(R, C, generator=g, device="cuda") < 0.001] *= 2.0 ** 10
    else:
        x[torch.rand(R, C, generator=g, device="cuda") < 0.33] = 5.0
    t = us(x, gy)
    assert t <= 1.5 * base, (t, base)


@pytest.mark.parametrize("N,factor", [(300, 1.35), (512, 2.0), (600, 2.0)])
def test_time_of_large_tables(pwl, N, factor):
    # beyond the sizes that two cells per knot leave 16 channels (257 intervals) or 8 (517)
    C, R = 1024, 65536
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn(R, C, generator=g, device="cuda").clamp_(-1.99, 2.99)
    gy = torch.randn(R, C, generator=g, device="cuda")
    gx = torch.empty_like(x)

    def us(n):
        knots, values = (torch.tensor(a, device="cuda") for a in _tables(C, n))
        gv, gk = torch.zeros_like(values), torch.zeros_like(knots)
        times = []
        for _ in range(8):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            pwl.pwl_channels_backward(knots, values, x, gy, gx, gv, gk)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) * 1e3)
        return sorted(times)[3]

    t, base = us(N), us(256)
    assert t <= factor * base, (t, base)
