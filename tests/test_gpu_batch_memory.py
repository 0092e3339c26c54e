"""Device memory of a batch: slopes and cells of the knots (8 bytes per knot) are
held only by batches whose index is built through global memory."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_bytes_per_knot():
    import paper_1510_02975_gb300 as pwl
    from paper_1510_02975_gb300 import _build
    _build.build()
    f = {"kind": "gaussian", "a": -4.0, "b": 4.0, "p": [1.0, 0.0, 1.0]}
    n, functions = 4095, 1024
    pwl.Batch([f], [n], m_per_interval=1, cells_per_knot=1).close()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    b = pwl.Batch([f] * functions, [n] * functions, m_per_interval=1, cells_per_knot=1)
    used = free - torch.cuda.mem_get_info()[0]
    cells = b.info()["total_cells"]
    # FP64 knots and values 16, projection 48, FP32 knots and values 8, side records 16,
    # densities 8 and their chunk sums 24 per 256; 8 per cell
    knots = (n + 1) * functions
    assert used <= 97 * knots + 8 * cells + (4 << 20), (used, knots, cells)
