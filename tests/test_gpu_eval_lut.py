"""16-bit queries on streams long enough for the table of all 65536 values:
the same bits as short streams (which go through the index) on every pattern,
for every index layout, aligned or not, and after an in-place update."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

M = 1 << 25


@pytest.fixture(scope="module")
def pwl():
    import paper_1510_02975_gb300 as m
    from paper_1510_02975_gb300 import _build
    _build.build()
    return m


def _table(pwl, kind, n, k_cells, values):
    f = {"gaussian": {"kind": "gaussian", "a": -4.0, "b": 4.0, "p": [1.0, 0.0, 1.0]},
         "lorentzian": {"kind": "lorentzian", "a": -10.0, "b": 10.0, "p": [1.0, 0.0, 1.0]}}[kind]
    k = pwl.pwl_design(f, n)
    return pwl.Table(k, pwl.pwl_project(f, k), values, k_cells), k


def _same(pwl, t, dtype, offset):
    patterns = torch.arange(65536, dtype=torch.int32, device="cuda").to(torch.int16).view(dtype)
    want = t(patterns).view(torch.int16)
    buf = torch.empty(M + 65536 + offset, dtype=dtype, device="cuda")
    m = M + 4321
    x = buf[offset:offset + m]
    x.view(torch.int16).copy_(patterns.view(torch.int16).repeat(m // 65536 + 1)[:m])
    y = t(x).view(torch.int16)
    assert torch.equal(y, want.repeat(m // 65536 + 1)[:m])
    t(x, x)  # in place
    assert torch.equal(x.view(torch.int16), y)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "fp16"])
@pytest.mark.parametrize("kind,n,k_cells,layout", [("gaussian", 1, 0, 0), ("gaussian", 256, 0, 0),
                                                   ("lorentzian", 4096, 0, 2), ("gaussian", 700, 300, 1)])
def test_long_streams_match_short_ones(pwl, kind, n, k_cells, layout, dtype):
    t, _ = _table(pwl, kind, n, k_cells, "fp32")
    assert t.info["layout"] == layout
    _same(pwl, t, dtype, 0)


@pytest.mark.parametrize("offset", [1, 3])
def test_unaligned_streams(pwl, offset):
    t, _ = _table(pwl, "gaussian", 64, 0, "bf16")
    _same(pwl, t, torch.bfloat16, offset)


def test_after_an_update(pwl):
    t, k = _table(pwl, "gaussian", 128, 0, "fp32")
    k2 = k.clone()
    k2[40:44] = k2[40] + torch.arange(4, device="cuda", dtype=torch.float64) * 1e-4  # several knots in a cell
    t.update(k2, torch.sin(k2))
    _same(pwl, t, torch.bfloat16, 0)
