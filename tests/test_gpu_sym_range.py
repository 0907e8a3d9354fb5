"""Symmetric polynomials with interfaces far thinner than the grid, or a tiny regularisation: products
of the raw-difference form's constants would leave FP32's range (a flat voxel then gave 0 times
infinity), so the general form runs.  Against the FP64 oracle: 1e-4 of the energy, 1e-3 of the
gradient's 2-norm (FP32 parity), and absolute values far below any that a curved field has where the
field is flat."""
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
SHAPE = (6, 24, 40)


@pytest.mark.parametrize("well", [0, 1])
@pytest.mark.parametrize("amp", [0.0, 0.1])
@pytest.mark.parametrize("eps, h, xi", [(1e-5, 1.0, 1e-15), (1e-10, 1.0, 1e-12), (1e-8, 1.0, 1e-4), (0.02, 0.01, 1e-13)])
def test_thin_interfaces(eps, h, xi, amp, well):
    u = I.noise(SHAPE, 0.3, amp, 3).astype(np.float32).astype(np.float64)
    Eo, go = oracle.energy_and_grad(u, {"a": SYM, "eps": eps, "h": h, "xi": xi, "well": well})
    ctx = pfc.Context(pfc.Problem.from_shape(SHAPE, eps=eps, h=h, a=SYM, xi=xi, well=well))
    ud = torch.tensor(u, dtype=torch.float32, device="cuda")
    E, g = ctx.energy_and_grad(ud)
    g = g.double().cpu().numpy()
    assert abs(E - Eo) <= 1e-4 * abs(Eo) + 1e-15
    assert abs(ctx.energy(ud) - Eo) <= 1e-4 * abs(Eo) + 1e-15
    assert np.linalg.norm(g - go) <= 1e-3 * np.linalg.norm(go) + 1e-15
    ctx.close()
