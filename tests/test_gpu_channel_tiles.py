"""The channel-wise kernels at the edges of their tiles (16, 8 and 4 channels
wide by table size), passes and flushes, over gradients of any magnitude, and
the BF16 backward against the FP32 one: parity with the oracle per channel."""
import numpy as np
import pytest

import oracle
from pwl_testutil import EVAL_REL, GRAD_REL

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pwl():
    import paper_1510_02975_gb300 as m
    from paper_1510_02975_gb300 import _build
    _build.build()
    return m


def _tables(C, N, seed):
    rng = np.random.default_rng(seed)
    base = np.linspace(-2.0, 3.0, N + 1)
    knots = np.tile(base, (C, 1))
    knots[:, 1:-1] += rng.uniform(-0.45, 0.45, (C, N - 1)) * (5.0 / N)
    return knots.astype(np.float32), rng.normal(size=(C, N + 1)).astype(np.float32)


def _cuda(*arrays):
    return [torch.tensor(a, device="cuda") for a in arrays]


def _check(pwl, knots, values, x, gy, k_cells=0, rows_per_bin=True):
    kt, vt = _cuda(knots, values)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    y = pwl.pwl_channels_forward(kt, vt, x, k_cells=k_cells, status=st).cpu().numpy().astype(np.float64)
    gv, gk = torch.zeros_like(vt), torch.zeros_like(kt)
    gx = pwl.pwl_channels_backward(kt, vt, x, gy, None, gv, gk, k_cells=k_cells, status=st).cpu().numpy()
    assert int(st.item()) == 0
    gv, gk = gv.cpu().numpy(), gk.cpu().numpy()
    xs, gs = x.cpu().numpy().astype(np.float64), gy.cpu().numpy().astype(np.float64)
    for c in range(knots.shape[0]):
        k, v = knots[c].astype(np.float64), values[c].astype(np.float64)
        r = oracle.evaluate(k, v, xs[:, c])
        assert np.abs(y[:, c] - r).max() <= EVAL_REL * np.abs(v).max(), c
        rgx, rgv, rgk, rva, rka = oracle.evaluate_grad(k, v, xs[:, c], gs[:, c])
        assert np.all(np.abs(gx[:, c] - rgx) <= EVAL_REL * np.abs(rgx) + 1e-30), c
        if rows_per_bin:
            assert np.all(np.abs(gv[c] - rgv) <= GRAD_REL * rva + 1e-30), c
            assert np.all(np.abs(gk[c] - rgk) <= GRAD_REL * rka + 1e-30), c
        else:  # bins of one or two elements: delta carries ulp(x) / h, which the sums do not
            assert abs(gv[c].sum(dtype=np.float64) - gs[:, c].sum()) <= GRAD_REL * np.abs(gs[:, c]).sum(), c
            assert abs(gk[c].sum(dtype=np.float64) + rgx.sum()) <= GRAD_REL * np.abs(rgx).sum() + 1e-30, c


def _x(R, C, knots, seed=1):
    x = torch.randn(R, C, generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda") * 1.5 + 0.5
    for r, j in enumerate((0, knots.shape[1] - 1, knots.shape[1] // 2)):  # both ends and a knot, exactly
        if r < R:
            x[r] = torch.tensor(knots[:, j], device="cuda")
    return x


@pytest.mark.parametrize("N", [1, 2, 3, 16])
@pytest.mark.parametrize("C,R", [(1, 1), (16, 63), (17, 64), (33, 65), (15, 1025), (32, 4097)])
def test_tile_and_pass_edges(pwl, C, R, N):
    knots, values = _tables(C, N, 10 * N + C)
    x = _x(R, C, knots)
    gy = torch.randn(R, C, generator=torch.Generator(device="cuda").manual_seed(2), device="cuda")
    _check(pwl, knots, values, x, gy, rows_per_bin=N < 16 or R > 4000)


@pytest.mark.parametrize("N", [255, 256, 257, 390, 512, 640])
def test_every_tile_width(pwl, N):
    C, R = 37, 700
    knots, values = _tables(C, N, N)
    x = _x(R, C, knots)
    gy = torch.randn(R, C, generator=torch.Generator(device="cuda").manual_seed(3), device="cuda")
    _check(pwl, knots, values, x, gy, rows_per_bin=False)


@pytest.mark.parametrize("k_cells", [1, 2, 7, 1200])
def test_requested_cells(pwl, k_cells):
    knots, values = _tables(19, 40, 5)
    x = _x(3000, 19, knots)
    gy = torch.randn(3000, 19, generator=torch.Generator(device="cuda").manual_seed(4), device="cuda")
    _check(pwl, knots, values, x, gy, k_cells=k_cells)


def test_more_rows_than_one_flush(pwl):
    # 8192 passes' worth of rows in one tile: the sums are flushed every 32512 rows
    C, N, R = 3, 4, 100001
    knots, values = _tables(C, N, 6)
    x = _x(R, C, knots)
    gy = torch.ones(R, C, device="cuda") * 0.7  # one sign: the words grow as fast as they can
    _check(pwl, knots, values, x, gy)


@pytest.mark.parametrize("case", ["1e-30", "1e25", "spread", "mostly_zero", "channels", "zero"])
def test_gradient_magnitudes(pwl, case):
    C, N, R = 20, 6, 6000
    knots, values = _tables(C, N, 7)
    x = _x(R, C, knots)
    g = torch.Generator(device="cuda").manual_seed(8)
    gy = torch.randn(R, C, generator=g, device="cuda")
    if case in ("1e-30", "1e25"):
        gy *= float(case)
    elif case == "spread":  # |gy| over 24 decades: most terms leave the fixed-point range or vanish in it
        gy *= 10.0 ** (torch.rand(R, C, generator=g, device="cuda") * 24 - 12)
    elif case == "mostly_zero":  # no sampled row of most channels is nonzero
        gy *= (torch.rand(R, C, generator=g, device="cuda") < 0.01) * 1e-6
    elif case == "channels":  # each channel its own magnitude
        gy *= 10.0 ** torch.linspace(-20, 20, C, device="cuda")
    else:
        gy.zero_()
    _check(pwl, knots, values, x, gy)


def test_nonfinite_gradients_stay_in_their_bins(pwl):
    C, N, R = 16, 8, 2000
    knots, values = _tables(C, N, 9)
    x = _x(R, C, knots)
    gy = torch.randn(R, C, generator=torch.Generator(device="cuda").manual_seed(5), device="cuda")
    kt, vt = _cuda(knots, values)
    gv0, gk0, gv, gk = (torch.zeros_like(vt) for _ in range(4))
    pwl.pwl_channels_backward(kt, vt, x, gy, None, gv0, gk0)
    mid = 0.5 * (knots[5, 3] + knots[5, 4])
    x[100, 5] = float(mid)
    gy[100, 5] = float("inf")
    x[200, 9] = float("nan")
    gx = pwl.pwl_channels_backward(kt, vt, x, gy, None, gv, gk)
    bad = torch.zeros_like(gv, dtype=torch.bool)
    bad[5, 3:5] = True
    assert torch.equal(~torch.isfinite(gv), bad) and torch.equal(~torch.isfinite(gk), bad)
    assert bool(torch.isnan(gx[200, 9])) and bool(torch.isinf(gx[100, 5]))
    others = [c for c in range(C) if c not in (5, 9)]
    assert torch.allclose(gv[others], gv0[others], rtol=1e-5, atol=1e-5)


def test_no_table_gradients_wanted(pwl):
    knots, values = _tables(17, 12, 3)
    kt, vt = _cuda(knots, values)
    x = _x(500, 17, knots)
    gy = torch.full((500, 17), 1e20, device="cuda")
    gy[::5] = 1.0
    gv, gk = torch.zeros_like(vt), torch.zeros_like(kt)
    gx = pwl.pwl_channels_backward(kt, vt, x, gy, None, gv, gk)
    assert torch.equal(gx, pwl.pwl_channels_backward(kt, vt, x, gy, None, None, None))
    gk2 = torch.zeros_like(kt)
    pwl.pwl_channels_backward(kt, vt, x, gy, None, None, gk2)
    assert torch.allclose(gk2, gk, rtol=1e-5, atol=1e-5 * float(gk.abs().max()))


@pytest.mark.parametrize("C,N,R", [(40, 256, 3001), (9, 31, 257), (16, 400, 600)])
def test_bf16_backward_is_the_fp32_one_on_widened_inputs(pwl, C, N, R):
    knots, values = _tables(C, N, N)
    kt, vt = _cuda(knots, values)
    x = _x(R, C, knots).to(torch.bfloat16)
    gy = torch.randn(R, C, generator=torch.Generator(device="cuda").manual_seed(6), device="cuda").to(torch.bfloat16)
    out = []
    for fn, xi, gi in ((pwl.pwl_channels_backward_bf16, x, gy), (pwl.pwl_channels_backward, x.float(), gy.float())):
        gv, gk = torch.zeros_like(vt), torch.zeros_like(kt)
        out.append((fn(kt, vt, xi, gi, None, gv, gk), gv, gk))
    assert torch.equal(out[0][0], out[1][0].to(torch.bfloat16))
    for a, b in zip(out[0][1:], out[1][1:]):  # the CTAs' sums are added in any order
        assert torch.allclose(a, b, rtol=1e-5, atol=1e-5 * float(b.abs().max()))


def test_unsorted_and_nonfinite_knots_are_flagged_and_stay_in_range(pwl):
    C, N, R = 20, 30, 2000
    knots, values = _tables(C, N, 11)
    good = _x(R, C, knots)
    gy = torch.ones(R, C, device="cuda")
    ref = pwl.pwl_channels_forward(*_cuda(knots, values), good)
    knots[3] = knots[3, ::-1]
    knots[4, 5] = np.nan
    knots[17, 0] = np.nan
    knots[18, 1:] = knots[18, 0]
    kt, vt = _cuda(knots, values)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    y = pwl.pwl_channels_forward(kt, vt, good, status=st)
    assert int(st.item()) & 1
    others = [c for c in range(C) if c not in (3, 4, 17, 18)]
    assert torch.equal(y[:, others], ref[:, others])
    st.zero_()
    pwl.pwl_channels_backward(kt, vt, good, gy, None, torch.zeros_like(vt), torch.zeros_like(kt), status=st)
    torch.cuda.synchronize()
    assert int(st.item()) & 1
