"""A source whose imaginary part is not finite at one node: the period's start takes the real part only, so
after two steps the displacement is not finite at that node alone (its neighbours take it up a step later,
through the stencil), in every precision, dimension and order."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1903_12522_gb300 import cmcg  # noqa: E402


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
@pytest.mark.parametrize("precision", [cmcg.FP64, cmcg.FP32, cmcg.MIXED])
@pytest.mark.parametrize("n,order", [((20, 17), 2), ((20, 17), 4), ((900, 800), 2), ((12, 13, 14), 2), ((12, 13, 14), 4)])
def test_imaginary_part(n, order, precision, bad):
    h = 1.0 / max(n)
    shape = tuple(m + 1 for m in reversed(n))
    dt = 0.2 * h
    s = cmcg.Solver(n, h, torch.ones(shape, dtype=torch.float64, device="cuda"), 2 * math.pi / (2 * dt), (0,) * 6,
                    precision=precision, order=order, dt=dt)
    assert s.info["steps_per_period"] == 2
    f = torch.zeros(shape, dtype=torch.complex128, device="cuda")
    at = tuple(m // 2 for m in shape)
    torch.view_as_real(f)[at][1] = bad
    y = torch.ones(shape, dtype=torch.float64, device="cuda")
    u, _ = s.wave_period(y, y, f)
    where = (~torch.isfinite(u)).nonzero().tolist()
    assert where == [list(at)]
    s.close()
