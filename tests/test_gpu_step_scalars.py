"""The five scalars of a step of the packed FP32 sweep, each against its own bar (energy, mass, mean
gradient, max|g|, mean|g|), on the shapes whose tiles, schedule and partial sums have edges.

Bars: a thread adds at most about 60 planes in FP32 (2^-24 of the running sum each), the rest is
compensated or FP64, so the sums carry at most 60 * 2^-25 = 1.8e-6 of the sum of magnitudes: 1e-6 for
the mass (|u| about 0.4), 1e-5 of mean|g| for the mean gradient and mean|g| (with the gradient's own
rounding, which averages out), 1e-5 of the energy (a sum of positive terms rounded at about 1e-6
each), 1e-4 for max|g| (one voxel).  A lost or doubled row, column, plane or partial is at least one
voxel in the grid: on the smallest shapes far above the bars, on the largest 1 / 382200 of a sum, so
a tile's row (32 voxels) or a block's partial shows there."""
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
SHAPES = [(5, 20, 32), (4, 21, 35), (3, 27, 35), (2, 25, 65), (6, 41, 34), (64, 41, 101), (70, 42, 97), (60, 49, 130),
          (60, 55, 97), (70, 53, 65)]


def _bars(Eo, go):
    gmean = np.abs(go).mean()
    return np.array([1e-5 * abs(Eo), 1e-6, 1e-5 * gmean, 1e-4 * np.abs(go).max(), 1e-5 * gmean])


@pytest.mark.parametrize("a, well", [(GEN, 0), (SYM, 1), (GEN, 1), (SYM, 0)])
@pytest.mark.parametrize("shape", SHAPES)
def test_scalars(shape, a, well):
    u = I.noise(shape, 0.3 if well == 0 else -0.4, 0.1, 7).astype(np.float32).astype(np.float64)
    Eo, go = oracle.energy_and_grad(u, {"a": a, "eps": 1.5, "h": 1.0, "xi": 1e-2, "well": well})
    ref = np.array([Eo, u.mean(), go.mean(), np.abs(go).max(), np.abs(go).mean()])
    bars = _bars(Eo, go)
    assert (bars < 1e-2 * np.abs(ref)).all()          # zeros, or a few percent off, do not pass
    ud = torch.tensor(u, dtype=torch.float32, device="cuda")
    for tile_y in (0, 13, 8):
        ctx = pfc.Context(pfc.Problem.from_shape(shape, eps=1.5, a=a, xi=1e-2, well=well, tile_y=tile_y))
        sc = torch.zeros(5, dtype=torch.float64, device="cuda")
        ctx.step(ud, torch.empty_like(ud), TAU, sc)
        assert (np.abs(sc.cpu().numpy() - ref) <= bars).all()
        ctx.close()
