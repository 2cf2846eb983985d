"""FP32 and mixed solves with the exact Riesz map on grids whose steps run on padded rows: the padded fields
share the PCG's vectors, so the solve has to give the bits of the flat step kernels, which have none."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1903_12522_gb300 import cmcg  # noqa: E402


@pytest.mark.parametrize("precision", [cmcg.FP32, cmcg.MIXED])
@pytest.mark.parametrize("n,order", [((8, 5, 6), 4), ((31, 20, 17), 4), ((201, 150, 97), 2)])
def test_same_bits_as_flat_steps(n, order, precision):
    h = 1.0 / max(n)
    shape = tuple(m + 1 for m in reversed(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(12)
    c = 1 + 0.5 * torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)
    f = torch.randn(shape, generator=gen, device="cuda", dtype=torch.complex128) / h ** 2
    out = []
    for tile in ((0, 0, 0, 0), (16, 0, 0, 3)):
        s = cmcg.Solver(n, h, c, 2 * math.pi / (10 * h), (0,) * 6, precision=precision, order=order, tile=tile, dt=0.22 * h,
                        max_iter=4, runup_periods=1)
        u, st = s.solve(f, tol=1e-12)
        x, code = s.riesz(u.real.contiguous())
        out.append((u, x, *s.adjoint_period(u.real.contiguous(), x), s.solve(f, tol=1e-12)[0]))
        s.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
