"""The Riesz map as on a device that holds no cluster of 16 CTAs: levels past one CTA run as launches.  The
exact map's residual as in test_gpu_riesz_levels, for grids whose V-cycles take the cluster otherwise (its
first level the finest or a coarser one, ragged coarsening) and one that takes none; an FP32 solve with the
V-cycle as Riesz map gives the same bits either way."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle.grid import Discretization  # noqa: E402
from paper_1903_12522_gb300 import cmcg  # noqa: E402

SIZES = [(17, 20), (64, 64), (101, 86), (257, 300), (12, 9, 10), (33, 30, 29), (50, 47, 44), (90, 87, 40)]


@pytest.mark.parametrize("n", SIZES)
def test_residual(n):
    rng = np.random.Generator(np.random.PCG64(2))
    shape = tuple(m + 1 for m in reversed(n))
    h = 1.0 / max(n)
    omega, dt, c = 2 * np.pi / (10 * h), 0.4 * h / np.sqrt(len(n)), np.ones(shape)
    dz = Discretization(n, h, c, omega, (0,) * 6, dt)
    s = cmcg.Solver(n, h, c, omega, (0,) * 6, dt=dt)
    cmcg.cmcg_no_cluster_selftest(s.handle)
    rhs = rng.standard_normal(shape)
    rhs = rhs - rhs.sum() / dz.W.sum() * dz.W
    for _ in range(2):
        sol, code = s.riesz(rhs)
        assert code == cmcg.OK
        assert np.linalg.norm(dz.K(sol.cpu().numpy()) - rhs) <= 1e-10 * np.linalg.norm(rhs)
    s.close()


@pytest.mark.parametrize("n", SIZES)
def test_vcycle_solve_keeps_its_bits(n):
    h = 1.0 / max(n)
    shape = tuple(m + 1 for m in reversed(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(9)
    c = 1 + 0.3 * torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)
    f = torch.randn(shape, generator=gen, device="cuda", dtype=torch.complex128) / h ** 2
    out = []
    for clusters in (True, False):
        s = cmcg.Solver(n, h, c, 2 * math.pi / (12 * h), (0,) * 6, precision=cmcg.FP32, flags=cmcg.FLAG_INEXACT_RIESZ,
                        dt=0.25 * h, max_iter=5)
        if not clusters:
            cmcg.cmcg_no_cluster_selftest(s.handle)
        out.append(s.solve(f, tol=1e-12)[0])
        s.close()
    assert torch.equal(*out)
