"""16-bit queries on long streams through tables whose knots crowd into a cell
(spaced by the logarithm): the same bits as short streams, before and after an
update that moves knots together, and no slower per query than through the
FP32 index."""
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


def _log_knots(n, octaves=40):
    return torch.cat([torch.zeros(1, dtype=torch.float64), 2.0 ** torch.linspace(2 - octaves, 2, n, dtype=torch.float64)]).cuda()


def _same_as_short(t, dtype):
    patterns = torch.arange(65536, dtype=torch.int32, device="cuda").to(torch.int16)
    want = t(patterns.view(dtype)).view(torch.int16)
    y = t(patterns.repeat(M // 65536 + 1).view(dtype)).view(torch.int16)
    assert torch.equal(y, want.repeat(M // 65536 + 1))


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "fp16"])
@pytest.mark.parametrize("n,k_cells", [(4, 0), (8, 0), (16, 0), (600, 0), (4000, 0), (300, 300), (7, 8)])
def test_crowded_knots(pwl, n, k_cells, dtype):
    k = _log_knots(n)
    _same_as_short(pwl.Table(k, torch.log1p(k), "fp32", k_cells), dtype)


@pytest.mark.parametrize("n,k_cells", [(128, 0), (4096, 0), (700, 300)])
def test_crowded_by_an_update(pwl, n, k_cells):
    k = torch.linspace(0, 4, n + 1, dtype=torch.float64, device="cuda")
    t = pwl.Table(k, torch.log1p(k), "fp32", k_cells)
    k2 = _log_knots(n, 20)
    t.update(k2, torch.log1p(k2))
    _same_as_short(t, torch.bfloat16)


def _us(t, x):
    y = torch.empty_like(x)
    times = []
    for _ in range(8):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        t(x, y)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b) * 1e3)
    return sorted(times)[3]


@pytest.mark.parametrize("n", [512, 2048, 8192])
def test_time_on_crowded_knots(pwl, n):
    # one query fewer goes through the index
    k = _log_knots(n)
    t = pwl.Table(k, torch.log1p(k))
    x = (torch.rand(M, device="cuda") * 4).bfloat16()
    long, short = _us(t, x), _us(t, x[:-1])
    assert long <= 1.2 * short, (long, short)
