"""J at the result of an FP32 or mixed solve, an FP64 period outside the handle's precision: with the
iteration stopped at the zero guess it is the J of the zero guess that an FP64 handle reports (1e-12:
sums of squares of FP64 periods).  2D grids with and without an on-chip loop, and 3D, both orders."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1903_12522_gb300 import cmcg  # noqa: E402


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("n", [(16, 9), (130, 61), (700, 300), (1500, 900), (13, 12, 17), (64, 40, 33)])
def test_J_of_the_zero_guess(n, order):
    h = 1.0 / max(n)
    shape = tuple(m + 1 for m in reversed(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(9)
    c = 1 + 0.3 * torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)
    f = torch.randn(shape, generator=gen, device="cuda", dtype=torch.complex128)
    faces = (cmcg.BC_ABC,) * (2 * len(n)) + (cmcg.BC_NEUMANN,) * (6 - 2 * len(n))

    def solve(precision):
        s = cmcg.Solver(n, h, c, 2 * math.pi / (12 * h), faces, precision=precision, order=order, dt=0.2 * h,
                        flags=0 if precision == cmcg.FP64 else cmcg.FLAG_INEXACT_RIESZ)
        st = [s.solve(f, g, tol=2.0)[1] for g in (None, f)]
        s.close()
        return st

    ref = solve(cmcg.FP64)
    for precision in (cmcg.FP32, cmcg.MIXED):
        for a, b in zip(solve(precision), ref):
            assert a["iterations"] == 0
            assert abs(a["J_final"] - b["J0"]) <= 1e-12 * b["J0"]
