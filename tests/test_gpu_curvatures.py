"""FP64 curvatures: bound by FP64 roots and quotients, so a thread per voxel.  One call on a 16^3 grid
takes under 20 us with its host part, and 69 us where each thread works through eight planes; 40 us
is between the two.  Values against the oracle on grids with partial blocks."""
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

A = (1.0, 0.0, 1.0, 0.0, 0.0, 0.0)


def test_small_grids_do_not_wait_for_a_march():
    shape = (16, 16, 16)
    ctx = pfc.Context(pfc.Problem.from_shape(shape, eps=1.5, a=A, well=1, prec="fp64"))
    u = torch.tensor(I.noise(shape, 0.0, 0.3, 1), device="cuda")
    took = []
    for _ in range(9):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        for _ in range(50):
            ctx.curvatures(u)
        b.record()
        torch.cuda.synchronize()
        took.append(a.elapsed_time(b) / 50 * 1e3)
    assert np.median(took) < 40.0
    ctx.close()


@pytest.mark.parametrize("proj", [0, 1])
@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 5, 17), (7, 9, 11), (40, 41, 43)])
def test_values(shape, proj):
    """xi = 1e-2: nothing sits at the kink of the root; 1e-9 of the largest curvature."""
    u = I.noise(shape, 0.0, 0.3, 2)
    op = {"a": A, "eps": 1.5, "h": 1.0, "xi": 1e-2, "well": 1, "proj": proj}
    want = oracle.curvatures(u, op)
    ctx = pfc.Context(pfc.Problem.from_shape(shape, eps=1.5, a=A, xi=1e-2, well=1, prec="fp64", proj=proj))
    got = ctx.curvatures(torch.tensor(u, device="cuda"))
    for g, w in zip(got, want):
        assert np.abs(g.cpu().numpy() - w).max() <= 1e-9 * max(np.abs(w).max(), 1e-12)
    ctx.close()
