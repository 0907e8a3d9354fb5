"""Edges of the curvature-diagram kernels: the two corner-mask paths (rows of a multiple of four
values on an aligned field, and any other), chunk and row ends, the count alone against the records,
short outputs, and the histogram's binning at bin edges, out of range and for non-finite values.

The records are compared bit for bit between the two paths (they differ only in how the corners are
read).  The histogram is compared with a FP64 one: bins exactly, sums to 1e-13 of the total weight
(FP64 additions in another order)."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="needs a GPU")]
else:
    pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_2103_04856_gb300 import pfc  # noqa: E402


def _field(shape, seed):
    rng = np.random.default_rng(seed)
    return rng.standard_normal(shape).astype(np.float32)


@pytest.mark.parametrize("shape", [(1, 1, 4), (2, 3, 8), (5, 7, 12), (9, 17, 100), (16, 16, 16), (3, 2, 1028)])
def test_mask_paths_agree(shape):
    """The same field on a 16-byte boundary and 4 bytes past one."""
    u = _field(shape, 1)
    n = u.size
    raw = torch.empty(n + 4, device="cuda")
    odd = raw[1:1 + n].view(shape)
    odd.copy_(torch.tensor(u))
    even = torch.tensor(u, device="cuda")
    assert odd.data_ptr() % 16 == 4 and even.data_ptr() % 16 == 0
    ctx = pfc.Context(pfc.Problem.from_shape(shape, eps=1.5, a=(1, 0, 1, 0, 0, 0), well=1))
    a, b = ctx.surface_cells(even, 0.1), ctx.surface_cells(odd, 0.1)
    assert a.shape[0] > 0 and torch.equal(a.view(torch.int32), b.view(torch.int32))
    ctx.close()


@pytest.mark.parametrize("shape", [(3, 5, 7), (4, 4, 257), (11, 13, 31), (8, 16, 64)])
def test_records_against_the_oracle(shape):
    u = _field(shape, 2)
    want = oracle.surface_cells(u.astype(np.float64), {"a": (1.0, 0, 1.0, 0, 0, 0), "eps": 1.5, "h": 1.0,
                                                       "xi": 1e-6, "well": 1}, 0.1)
    ctx = pfc.Context(pfc.Problem.from_shape(shape, eps=1.5, a=(1, 0, 1, 0, 0, 0), well=1, prec="fp64"))
    ud = torch.tensor(u, dtype=torch.float64, device="cuda")
    got = ctx.surface_cells(ud, 0.1).cpu().numpy()
    assert got.shape == want.shape
    assert np.allclose(got[:, 0], want[:, 0], rtol=1e-11, atol=1e-13)
    # a short output: the first records and the full count
    lib, n, cap = pfc.load_library(), ctypes.c_int64(), max(1, got.shape[0] // 2)
    out = torch.full((cap + 1, 3), -7.0, dtype=torch.float64, device="cuda")
    assert lib.pfc_surface_cells(ctx._h, ctypes.c_void_p(ud.data_ptr()), 0.1, ctypes.c_void_p(out.data_ptr()), cap,
                                 ctypes.byref(n), None) == 0
    assert n.value == got.shape[0]
    assert np.array_equal(out[:cap].cpu().numpy(), got[:cap]) and bool((out[cap] == -7.0).all())
    ctx.close()


@pytest.mark.parametrize("nbins, lo, hi", [(1, -1.0, 1.0), (100, -2.0, 2.0), (100, 1000.0, 1001.0), (37, -1e-3, 3e-3),
                                           (1500, -100.0, 100.0)])
def test_histogram_bins(nbins, lo, hi):
    """(1500 bins take one table, the others a table per SM.)"""
    rng = np.random.default_rng(nbins)
    n = 20000
    c = rng.uniform(lo - 0.1 * (hi - lo), hi + 0.1 * (hi - lo), (n, 3)).astype(np.float32)
    c[:4000, 1:] = (lo + (hi - lo) / nbins * rng.integers(-2, nbins + 3, (4000, 2))).astype(np.float32)   # bin edges
    c[:, 0] = rng.uniform(0.0, 1.0, n).astype(np.float32)
    c[4000:4006, 1] = [np.inf, -np.inf, np.nan, 3e38, -3e38, 0.0]
    x = c.astype(np.float64)
    with np.errstate(over="ignore"):
        b = np.floor((np.nan_to_num(x[:, 1:], nan=lo) - lo) * (nbins / (hi - lo)))
    b = np.clip(b, 0, nbins - 1).astype(np.int64)
    want = np.zeros((nbins, nbins))
    np.add.at(want, (b[:, 0], b[:, 1]), x[:, 0])
    ctx = pfc.Context(pfc.Problem.from_shape((4, 4, 4), eps=1.5, a=(1, 0, 1, 0, 0, 0)))
    for _ in range(2):
        got = ctx.curvature_histogram(torch.tensor(c, device="cuda"), nbins, lo, hi).cpu().numpy()
        assert np.array_equal(got != 0, want != 0)
        assert np.abs(got - want).max() <= 1e-13 * x[:, 0].sum()
    ctx.close()


@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 3, 5), (17, 9, 33), (25, 8, 64)])
def test_curvatures_edges(shape):
    """The marching kernel's chunk, row and column ends, FP32 against FP64 on the same field: k1 and k2
    to 1e-3 of their scale (FP32 cancellation in D is the larger part of that)."""
    u = _field(shape, 5)
    k = {}
    for prec in ("fp64", "fp32"):
        p = pfc.Problem.from_shape(shape, eps=1.5, a=(1, 0, 1, 0, 0, 0), well=1, prec=prec)
        ctx = pfc.Context(p)
        k[prec] = [t.double().cpu().numpy() for t in ctx.curvatures(torch.tensor(u, dtype=p.dtype, device="cuda"))]
        ctx.close()
    o = oracle.curvatures(u.astype(np.float64), {"a": (1.0, 0, 1.0, 0, 0, 0), "eps": 1.5, "h": 1.0, "xi": 1e-6, "well": 1})
    for j in range(2):
        scale = np.abs(o[j]).max() + 1e-12
        assert np.abs(k["fp64"][j] - o[j]).max() <= 1e-6 * scale
        assert np.abs(k["fp32"][j] - k["fp64"][j]).max() <= 1e-3 * scale
