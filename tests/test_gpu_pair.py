"""The packed FP32 sweep (two rows per thread, tiles of 20, 12 or 8 rows, 24 for
the energy alone) at the sizes where its tiles, warps and schedule have edges:
ragged last rows of tiles of every kind, rows shorter than a tile or not a
multiple of a 16-byte load, runs of one plane, and enough planes per CTA for the
weighted schedule; energy, gradient and step, both forms of the polynomial and
both double wells, against the FP64 oracle.

Bars: xi = 1e-2, so no voxel sits at a kink narrower than FP32 resolves; the
density is a sum of about 30 products of the field's second differences, each
rounded at 6e-8, and the gradient of second differences of those: 1e-5 of the
energy and 1e-4 of the gradient's 2-norm and of max|g| leave a factor of ten,
where a wrong row, column or plane shows at O(1).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="needs a GPU")]
else:
    pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_2103_04856_gb300 import inputs as I  # noqa: E402
from paper_2103_04856_gb300 import pfc  # noqa: E402

SYM = (1.0, 0.4, 1.0, 0.3, 0.3, -0.2)
GEN = (0.8, 0.3, 1.1, 0.4, -0.2, 0.1)
TAU = 1e-3
# (nz, ny, nx): one row and column; a tile and its edges in y; pairs cut in two by the ragged
# edge; 24-row energy tiles and theirs; rows of 31-33 and of no 16-byte multiple; and a grid of
# more than four planes per CTA whose last tiles hold one, two or nine rows
SHAPES = [(3, 1, 1), (1, 2, 33), (2, 19, 31), (5, 20, 32), (4, 21, 35), (3, 24, 30), (2, 25, 65), (6, 41, 34),
          (64, 41, 101), (70, 42, 97), (60, 49, 130)]


def _cmp(shape, a, well, tile_y):
    u = I.noise(shape, 0.3 if well == 0 else -0.4, 0.1, 7).astype(np.float32).astype(np.float64)
    op = {"a": a, "eps": 1.5, "h": 1.0, "xi": 1e-2, "well": well}
    Eo, go = oracle.energy_and_grad(u, op)
    uo, _ = oracle.step(u, op, TAU)
    ctx = pfc.Context(pfc.Problem.from_shape(shape, eps=1.5, a=a, xi=1e-2, well=well, tile_y=tile_y))
    ud = torch.tensor(u, dtype=torch.float32, device="cuda")
    E, g = ctx.energy_and_grad(ud)
    g = g.double().cpu().numpy()
    gmax = np.abs(go).max()
    assert abs(E - Eo) <= 1e-5 * max(abs(Eo), 1e-3 * u.size)
    assert abs(ctx.energy(ud) - Eo) <= 1e-5 * max(abs(Eo), 1e-3 * u.size)
    assert np.linalg.norm(g - go) <= 1e-4 * np.linalg.norm(go) + 1e-7 * np.sqrt(u.size)
    assert np.abs(g - go).max() <= 1e-4 * gmax + 1e-7
    out = torch.empty_like(ud)
    sc = torch.zeros(5, dtype=torch.float64, device="cuda")
    ctx.step(ud, out, TAU, sc)
    assert np.abs(out.double().cpu().numpy() - uo).max() <= 2.0 ** -23 + TAU * (1e-4 * gmax + 1e-7)
    sc = sc.cpu().numpy()
    ref = np.array([Eo, u.mean(), go.mean(), gmax, np.abs(go).mean()])
    assert np.abs(sc - ref).max() <= 1e-5 * max(abs(Eo), 1e-3 * u.size) + 1e-4 * gmax
    ctx.close()


@pytest.mark.parametrize("tile_y", [0, 13, 8])
@pytest.mark.parametrize("shape", SHAPES)
def test_packed_sweep_edges(shape, tile_y):
    _cmp(shape, GEN, 0, tile_y)
    _cmp(shape, SYM, 1, tile_y)


@pytest.mark.parametrize("a, well", [(GEN, 1), (SYM, 0)])
def test_packed_sweep_other_wells(a, well):
    _cmp((64, 41, 101), a, well, 0)


def test_packed_batch_of_ragged_problems():
    """A batch whose problems differ in size, polynomial and double well: each as alone."""
    shapes = [(30, 41, 37), (50, 20, 66), (9, 61, 129), (64, 42, 33)]
    probs, us = [], []
    for k, s in enumerate(shapes):
        probs.append(pfc.Problem.from_shape(s, eps=1.5, a=(GEN, SYM)[k % 2], xi=1e-2, well=k // 2))
        us.append(torch.tensor(I.noise(s, 0.3, 0.1, k), dtype=torch.float32, device="cuda"))
    outs = [torch.empty_like(u) for u in us]
    b = pfc.Batch(probs)
    b.step(us, outs, TAU)
    for p, u, o in zip(probs, us, outs):
        alone = torch.empty_like(u)
        ctx = pfc.Context(p)
        ctx.step(u, alone, TAU)
        assert (o - alone).abs().max().item() <= 2.0 ** -22
        ctx.close()
    b.close()


def test_symmetric_constants_out_of_range_take_the_general_form():
    """xi so small that xi^2 / sg^2 is no FP32 number: the symmetric form's constants do not fit."""
    shape = (6, 21, 40)
    u = I.noise(shape, 0.3, 0.1, 3).astype(np.float32).astype(np.float64)
    op = {"a": SYM, "eps": 0.02, "h": 1e-3, "xi": 1e-17, "well": 0}
    Eo, go = oracle.energy_and_grad(u, op)
    ctx = pfc.Context(pfc.Problem.from_shape(shape, eps=0.02, h=1e-3, a=SYM, xi=1e-17))
    E, g = ctx.energy_and_grad(torch.tensor(u, dtype=torch.float32, device="cuda"))
    assert abs(E - Eo) <= 1e-4 * abs(Eo)
    assert np.linalg.norm(g.double().cpu().numpy() - go) <= 1e-3 * np.linalg.norm(go)
    ctx.close()


@pytest.mark.parametrize("nx", [30, 31, 32, 36, 65, 100])
@pytest.mark.parametrize("ny, nz", [(1, 3), (21, 2), (24, 5), (41, 40)])
def test_packed_extended_sweep_edges(nx, ny, nz):
    """Coefficients from a field with the orientation term: its planes travel in 16-byte pieces where
    nx is a multiple of four, else value by value; tiles ragged in both directions."""
    shape = (nz, ny, nx)
    u = I.noise(shape, 0.3, 0.1, 7).astype(np.float32).astype(np.float64)
    rng = np.random.default_rng(nx + ny)
    base = np.array(GEN)[:, None, None, None]
    af = (base * (1.0 + 0.3 * rng.standard_normal((6,) + shape))).astype(np.float32)
    mu, theta = 0.7, (0.6, 0.0, 0.8)
    op = {"a": GEN, "eps": 1.5, "h": 1.0, "xi": 1e-2, "well": 0, "mu": mu, "theta": theta, "a_field": af.astype(np.float64)}
    Eo, go = oracle.energy_and_grad(u, op)
    ctx = pfc.Context(pfc.Problem.from_shape(shape, eps=1.5, a=GEN, xi=1e-2, mu=mu, theta=theta))
    ctx.set_coefficient_field(torch.tensor(af, device="cuda"))
    ud = torch.tensor(u, dtype=torch.float32, device="cuda")
    E, g = ctx.energy_and_grad(ud)
    gmax = np.abs(go).max()
    assert abs(E - Eo) <= 1e-5 * max(abs(Eo), 1e-3 * u.size)
    assert abs(ctx.energy(ud) - Eo) <= 1e-5 * max(abs(Eo), 1e-3 * u.size)
    assert np.abs(g.double().cpu().numpy() - go).max() <= 1e-4 * gmax + 1e-7
    out = torch.empty_like(ud)
    ctx.step(ud, out, TAU)
    lam = go.mean()
    assert np.abs(out.double().cpu().numpy() - (u - TAU * (go - lam))).max() <= 2.0 ** -23 + TAU * (1e-4 * gmax + 1e-7)
    ctx.close()


@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 2, 3), (2, 3, 5), (32, 32, 32), (5, 40, 36)])
@pytest.mark.parametrize("a, well", [(SYM, 0), (SYM, 1), (GEN, 0), (GEN, 1)])
def test_fp64_two_kernel_form(shape, a, well):
    """The FP64 two-kernel evaluation against the oracle at 1e-10, and against the fused sweep (which an
    explicit tile height selects)."""
    u = I.noise(shape, 0.3, 0.1, 11)
    op = {"a": a, "eps": 1.5, "h": 1.0, "xi": 1e-2, "well": well}
    Eo, go = oracle.energy_and_grad(u, op)
    uo, _ = oracle.step(u, op, TAU)
    ud = torch.tensor(u, device="cuda")
    scale = max(np.abs(go).max(), 1e-3)
    res = []
    for tile_y in (0, 8):
        ctx = pfc.Context(pfc.Problem.from_shape(shape, eps=1.5, a=a, xi=1e-2, well=well, prec="fp64", tile_y=tile_y))
        E, g = ctx.energy_and_grad(ud)
        assert abs(E - Eo) <= 1e-10 * max(abs(Eo), 1e-6 * u.size)
        assert abs(ctx.energy(ud) - Eo) <= 1e-10 * max(abs(Eo), 1e-6 * u.size)
        assert np.abs(g.cpu().numpy() - go).max() <= 1e-10 * scale
        out = torch.empty_like(ud)
        sc = torch.zeros(5, dtype=torch.float64, device="cuda")
        ctx.step(ud, out, TAU, sc)
        assert np.abs(out.cpu().numpy() - uo).max() <= 1e-13
        res.append(sc.cpu().numpy())
        ctx.close()
    assert np.abs(res[0] - res[1]).max() <= 1e-10 * max(abs(Eo), scale)


@pytest.mark.parametrize("shape", [(3, 21, 31), (1, 26, 33), (4, 27, 35), (2, 28, 64), (60, 55, 97), (64, 56, 130),
                                   (70, 53, 65)])
def test_packed_tall_tiles(shape):
    """Heights at which symmetric polynomials take tiles of 28 rows (whole, and ragged by one to seven rows)."""
    _cmp(shape, SYM, 0, 0)


@pytest.mark.parametrize("a", [GEN, SYM])
@pytest.mark.parametrize("shape", [(3, 29, 31), (2, 30, 33), (5, 31, 64), (40, 61, 97)])
def test_packed_energy_tiles(shape, a):
    """The energy alone: heights around its tiles of 30 rows."""
    _cmp(shape, a, 1, 0)


def test_packed_batch_with_tall_tiles():
    """A batch of symmetric polynomials whose heights together ask for tiles of 28 rows: each as alone."""
    shapes = [(30, 56, 37), (50, 28, 66), (9, 27, 129), (64, 20, 33)]
    probs = [pfc.Problem.from_shape(s, eps=1.5, a=SYM, xi=1e-2, well=k % 2) for k, s in enumerate(shapes)]
    us = [torch.tensor(I.noise(s, 0.3, 0.1, k), dtype=torch.float32, device="cuda") for k, s in enumerate(shapes)]
    outs = [torch.empty_like(u) for u in us]
    b = pfc.Batch(probs)
    b.step(us, outs, TAU)
    for p, u, o in zip(probs, us, outs):
        alone = torch.empty_like(u)
        ctx = pfc.Context(p)
        ctx.step(u, alone, TAU)
        assert (o - alone).abs().max().item() <= 2.0 ** -22
        ctx.close()
    b.close()
