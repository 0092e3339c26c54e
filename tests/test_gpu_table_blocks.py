"""Table blocks are reused by later tables: results do not depend on what a
block held before, nor on streams and threads that build and destroy tables
at the same time."""
import threading

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

F = {"kind": "gaussian", "a": -4.0, "b": 4.0, "p": [1.0, 0.0, 1.0]}


@pytest.fixture(scope="module")
def pwl():
    import paper_1510_02975_gb300 as m
    from paper_1510_02975_gb300 import _build
    _build.build()
    return m


def _arrays(pwl, n):
    k = pwl.pwl_design(F, n)
    return k, pwl.pwl_project(F, k)


def test_alternating_sizes(pwl):
    x = torch.rand(100003, device="cuda") * 9 - 4.5
    sizes = [1, 63, 700, 64, 4096, 2, 9000]
    arrays = {n: _arrays(pwl, n) for n in sizes}
    keep = {n: pwl.Table(*arrays[n]) for n in sizes}
    want = {n: keep[n](x) for n in sizes}
    for _ in range(6):
        for n in sizes:
            t = pwl.Table(*arrays[n])
            y = t(x)
            t.close()  # with the evaluation in flight
            assert torch.equal(y, want[n]), n


def test_threads_with_their_own_streams(pwl):
    arrays = [_arrays(pwl, n) for n in (40, 300, 1000, 2000)]
    x = torch.rand(1 << 20, device="cuda") * 8 - 4
    want = [pwl.Table(*a)(x) for a in arrays]
    torch.cuda.synchronize()
    wrong = []

    def work(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(25):
                t = pwl.Table(*arrays[i])
                y = t(x)
                t.close()
                torch.cuda.current_stream().synchronize()
                if not torch.equal(y, want[i]):
                    wrong.append(i)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(arrays))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


@pytest.mark.parametrize("where, mode", [("here", "relaxed"), ("thread", "relaxed"), ("thread", "thread_local")])
@pytest.mark.parametrize("n", [63, 9000])
def test_destroying_leaves_a_capture_alone(pwl, where, mode, n):
    """A graph capture goes on while a table is destroyed, in any mode and thread that cudaFree
    allows, and so does one during which another thread builds, uses and destroys a table."""
    arrays = _arrays(pwl, n)
    kept, gone = pwl.Table(*arrays), pwl.Table(*arrays)
    x = torch.rand(100003, device="cuda") * 8 - 4
    want = kept(x)
    y, z = torch.empty_like(x), torch.empty_like(x)
    torch.cuda.synchronize()

    def destroy():
        gone.close()
        if where == "thread":
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(3):
                    t = pwl.Table(*arrays)
                    t(x, z)
                    t.close()

    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode=mode):
        kept(x, y)
        if where == "here":
            destroy()
        else:
            t = threading.Thread(target=destroy)
            t.start()
            t.join()
        y.add_(1.0)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, want + 1.0)
    assert where == "here" or torch.equal(z, want)
