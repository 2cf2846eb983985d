"""Grids with more z-planes than a launch has blocks along y at the kernels' usual planes per thread
(65535 blocks): FP32 steps on padded rows against the flat z-pair kernels (same bits), FP32 first-order
periods against FP64 ones (2e-5 relative L2, as against the oracle), and the Riesz map with ragged
coarsening (residual as in test_gpu_riesz_levels; every tenth plane is Dirichlet, so that it converges)."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle.grid import Discretization  # noqa: E402
from paper_1903_12522_gb300 import cmcg  # noqa: E402
from test_gpu_step_row import periods  # noqa: E402


@pytest.mark.parametrize("order", [2, 4])
def test_steps_on_padded_rows(order):
    n = (8, 2 if order == 2 else 4, 262200)
    for f, g in ((0, 0), (1, 1)):
        a = periods(n, order, (0,) * 6, (16, 0, 0, 3), f, g)
        b = periods(n, order, (0,) * 6, (0, 0, 0, 0), f, g)
        for x, y in zip(a, b):
            assert torch.equal(x, y)


def test_first_order_periods():
    n, shape = (2, 2, 131100), (131101, 3, 3)
    h = 0.01
    gen = torch.Generator(device="cuda")
    gen.manual_seed(8)

    def rnd(k):
        return torch.randn((k, *shape), generator=gen, device="cuda", dtype=torch.float64)

    s0, f, y = rnd(4).reshape(-1), torch.complex(rnd(1), rnd(1)).reshape(-1) / h, rnd(4).reshape(-1)
    c = 1.0 + torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)
    out = {}
    for precision in (cmcg.FP64, cmcg.FP32):
        s = cmcg.Solver(n, h, c, 2 * math.pi / (9 * h), (cmcg.BC_ABC,) * 6, precision=precision, dt=0.2 * h,
                        flags=cmcg.FLAG_FIRST_ORDER)
        out[precision] = s.fo_period(s0), s.fo_period(s0, f, f), s.fo_adjoint_period(y)
        s.close()
    for a, b in zip(out[cmcg.FP32], out[cmcg.FP64]):
        assert ((a - b).norm() <= 2e-5 * b.norm()).item()


def test_riesz_map_with_ragged_coarsening():
    n, shape = (5, 5, 131100), (131101, 6, 6)
    h = 1.0
    mask = np.zeros(shape, np.uint8)
    mask[::10] = 1
    c = np.ones(shape)
    dz = Discretization(n, h, c, 0.5, (0,) * 6, 0.4, mask=mask)
    s = cmcg.Solver(n, h, c, 0.5, (0,) * 6, mask=mask, dt=0.4)
    rhs = np.random.Generator(np.random.PCG64(2)).standard_normal(shape) * dz.act
    sol, code = s.riesz(rhs)
    assert code == cmcg.OK
    assert np.linalg.norm(dz.K(sol.cpu().numpy()) - rhs) <= 1e-10 * np.linalg.norm(rhs)
    s.close()
