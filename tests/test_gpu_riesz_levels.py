"""The exact Riesz map where the V-cycle's coarse end changes its shape: levels in one CTA, levels
spread over a cluster, grid-wide levels above them; nested and ragged coarsening; with and without
Dirichlet nodes; a right-hand side and a solution at 8-byte alignment.

The residual is formed by the oracle's stiffness matrix.  PCG stops at 1e-12 relative to ||rhs||; the
recursive residual drifts from the true one by rounding of K s, at most 10 2^-53 ||K|| ||s||, which for
these grids (cond <= 1e5) stays below 1e-10 ||rhs||.  A V-cycle that lost its coarse correction would
need more than 60 iterations (CMCG_NOT_CONVERGED)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle.grid import Discretization  # noqa: E402
from paper_1903_12522_gb300 import cmcg  # noqa: E402

SIZES = [(2, 2), (4, 4), (7, 9), (32, 32), (43, 45), (64, 64), (101, 86), (200, 170), (257, 300), (260, 5),
         (9, 300), (300, 9), (2, 2, 2), (4, 4, 4), (12, 9, 10), (16, 16, 16), (33, 30, 29), (34, 33, 32), (50, 47, 44),
         (90, 87, 40), (57, 63, 44)]


@pytest.mark.parametrize("obstacle", [False, True])
@pytest.mark.parametrize("n", SIZES)
def test_riesz_residual(n, obstacle):
    rng = np.random.Generator(np.random.PCG64(2))
    shape = tuple(m + 1 for m in reversed(n))
    h = 1.0 / max(n)
    mask = None
    if obstacle:
        mask = np.zeros(shape, np.uint8)
        mask[tuple(slice(s // 3, s // 2 + 1) for s in shape)] = 1
    omega, dt = 2 * np.pi / (10 * h), 0.4 * h / np.sqrt(len(n))
    c = np.ones(shape)
    dz = Discretization(n, h, c, omega, (0,) * 6, dt, mask=mask)
    s = cmcg.Solver(n, h, c, omega, (0,) * 6, mask=mask, dt=dt)
    rhs = rng.standard_normal(shape) * dz.act
    if not obstacle:
        rhs = rhs - rhs.sum() / dz.W.sum() * dz.W
    # 8-byte aligned input and output
    raw = torch.empty(2 * rhs.size + 3, dtype=torch.float64, device="cuda")
    b, x = raw[1:1 + rhs.size], raw[2 + rhs.size:2 + 2 * rhs.size]
    b.copy_(torch.as_tensor(rhs.ravel()))
    torch.cuda.synchronize()
    for _ in range(2):  # the second solve runs its first iterations without host checks
        assert cmcg.cmcg_riesz(s.handle, b, x) == cmcg.OK
        sol = x.cpu().numpy().reshape(shape)
        assert np.linalg.norm(dz.K(sol) - rhs) <= 1e-10 * np.linalg.norm(rhs)
    s.close()
