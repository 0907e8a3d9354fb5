"""The curvature histogram only enqueues work on the caller's stream: calls of one context on two
streams do not meet, a call can be captured (the context's first one too), and a captured call stays
valid whatever the context is asked for afterwards.  Sums against FP64 ones on the host: bins
exactly, 1e-13 of the total weight (FP64 additions in another order)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="needs a GPU")]
else:
    pytestmark = pytest.mark.gpu

from paper_2103_04856_gb300 import pfc  # noqa: E402

LO, HI = -2.0, 2.0


def _cells(n, seed):
    """Cells whose curvatures crowd into few bins, as those of a smooth surface do."""
    rng = np.random.default_rng(seed)
    c = rng.normal(0.0, 0.2, (n, 3)).astype(np.float32)
    c[:, 0] = rng.uniform(0.1, 1.0, n)
    return c


def _want(c, nbins):
    x = c.astype(np.float64)
    b = np.clip(np.floor((x[:, 1:] - LO) * (nbins / (HI - LO))), 0, nbins - 1).astype(np.int64)
    w = np.zeros((nbins, nbins))
    np.add.at(w, (b[:, 0], b[:, 1]), x[:, 0])
    return w


def _check(got, want):
    got = got.cpu().numpy()
    assert np.array_equal(got != 0, want != 0)
    assert np.abs(got - want).max() <= 1e-13 * want.sum()


def _context():
    return pfc.Context(pfc.Problem.from_shape((4, 4, 4), eps=1.5, a=(1, 0, 1, 0, 0, 0)))


@pytest.mark.parametrize("n", [3000, 400000])
def test_two_streams_of_one_context(n):
    ctx = _context()
    host = [_cells(n, k) for k in range(2)]
    dev = [torch.tensor(c, device="cuda") for c in host]
    streams = [torch.cuda.Stream() for _ in range(2)]
    bins = [(100, 64), (40, 200), (100, 100), (200, 20)]     # of the two streams, in turn
    torch.cuda.synchronize()
    got = []
    for _ in range(5):
        for pair in bins:
            for k, s in enumerate(streams):
                with torch.cuda.stream(s):
                    got.append((k, pair[k], ctx.curvature_histogram(dev[k], pair[k], LO, HI)))
    torch.cuda.synchronize()
    want = {(k, b): _want(host[k], b) for k, b in {(k, p[k]) for p in bins for k in range(2)}}
    for k, b, h in got:
        _check(h, want[(k, b)])
    ctx.close()


@pytest.mark.parametrize("n", [0, 3000, 400000])
def test_captured_first_call_and_larger_ones_between_replays(n):
    other = _context()                       # the kernels are loaded before the capture
    other.curvature_histogram(torch.tensor(_cells(400000, 1), device="cuda"), 100, LO, HI)
    other.curvature_histogram(torch.tensor(_cells(10, 1), device="cuda"), 1500, LO, HI)
    torch.cuda.synchronize()
    ctx = _context()
    first, second = _cells(n, 2), _cells(n, 3)
    cells = torch.tensor(first, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        hist = ctx.curvature_histogram(cells, 100, LO, HI)
    big = _cells(1000000, 4)                 # with tables of its own at 300 and 600 bins
    for nbins, host in ((300, first), (600, second)):
        _check(ctx.curvature_histogram(torch.tensor(big, device="cuda"), nbins, LO, HI), _want(big, nbins))
        cells.copy_(torch.tensor(host))
        graph.replay()
        torch.cuda.synchronize()
        _check(hist, _want(host, 100))
    ctx.close()
    other.close()
