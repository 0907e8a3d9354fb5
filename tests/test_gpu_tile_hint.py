"""The FP32 tile-height hint on launches of many planes per SM: smaller tiles are slower there, so every
hint takes the automatic height, which shows in the scalars (sums in the same order: equal bits).
Small launches follow it (test_gpu_pair.py)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="needs a GPU")]
else:
    pytestmark = pytest.mark.gpu

from paper_2103_04856_gb300 import inputs as I  # noqa: E402
from paper_2103_04856_gb300 import pfc  # noqa: E402

GEN = (0.8, 0.3, 1.1, 0.4, -0.2, 0.1)
SYM = (1.0, 0.4, 1.0, 0.3, 0.3, -0.2)


@pytest.mark.parametrize("a", [GEN, SYM])
@pytest.mark.parametrize("shape", [(100, 100, 100), (64, 133, 97)])
def test_hints_of_large_launches(shape, a):
    u = torch.tensor(I.noise(shape, 0.3, 0.1, 5), dtype=torch.float32, device="cuda")
    res = []
    for tile_y in (0, 8, 13, 16):
        ctx = pfc.Context(pfc.Problem.from_shape(shape, eps=1.5, a=a, xi=1e-2, tile_y=tile_y))
        sc = torch.zeros(5, dtype=torch.float64, device="cuda")
        out = ctx.step(u, torch.empty_like(u), 1e-4, sc)
        res.append((sc.cpu().numpy(), out.cpu().numpy()))
        ctx.close()
    for sc, out in res[1:]:
        assert np.array_equal(sc, res[0][0]) and np.array_equal(out, res[0][1])
