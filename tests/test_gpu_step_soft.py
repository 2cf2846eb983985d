"""FP64 periods with the integer stencil sum against the CPU oracle: the smallest grids, chunk and
block remainders, both orders, every face kind, sources on faces only and inside, and data so small
or large that the plain FP64 sum takes over.

Tolerance: a step rounds its sum, its two terms and its result, a few units of 2^-53 of the largest
amplitude, and N leapfrog steps add these up with weights up to N: 4 N^2 2^-53 <= 1e-12 for the
N <= 47 steps used here, relative to the largest value."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import wave  # noqa: E402
from oracle.grid import Discretization  # noqa: E402
from paper_1903_12522_gb300 import cmcg  # noqa: E402
from paper_1903_12522_gb300 import workloads as wl  # noqa: E402

TOL = 1e-12
SIZES = [(2, 2), (2, 3), (15, 16), (40, 33), (2, 2, 2), (3, 2, 5), (16, 15, 8), (17, 16, 9), (33, 7, 31)]
FACES = [(0,) * 6, (0, 1, 2, 0, 1, 0)]


def problem(n, order, faces, seed):
    if order == 4:
        faces = tuple(1 if f == 2 else f for f in faces)  # the 4th-order stencil takes no Dirichlet nodes
    rng = np.random.Generator(np.random.PCG64(seed))
    shape = tuple(m + 1 for m in reversed(n))
    h = 1.0 / max(n)
    c = rng.uniform(1.0, 2.0, shape)
    omega = 2 * np.pi / (10 * h)
    dt = (0.9 if order == 2 else 0.75) * h / (2.0 * np.sqrt(len(n)))
    dz = Discretization(n, h, c, omega, faces, dt, order=order)
    assert dz.N <= 47
    s = cmcg.Solver(n, h, c, omega, faces, order=order, dt=dt)
    return dz, s, rng, shape


def close(got, ref):
    scale = max(np.abs(r).max() for r in ref)
    for a, b in zip(got, ref):
        assert np.abs(a.cpu().numpy() - b).max() <= TOL * scale


@pytest.mark.parametrize("faces", FACES)
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("n", SIZES)
def test_periods_match_oracle(n, order, faces):
    dz, s, rng, shape = problem(n, order, faces, 5)
    y, v = rng.standard_normal(shape), rng.standard_normal(shape) * dz.omega
    f = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    for src in ((None, None), (f * dz.omega ** 2, None), (None, f)):
        F = None if src[0] is None and src[1] is None else dz.load(*src)
        got = s.wave_period(y, v, *src)
        ref = wave.period(dz, y, v, F)
        close([got[0], got[1] / dz.omega], [ref[0], ref[1] / dz.omega])
    got, ref = s.adjoint_period(y, v), wave.transposed_period(dz, y, v)
    close(got, ref)
    s.close()


@pytest.mark.parametrize("scale", [1e-306, 1e-290, 1e-200, 1e250, 1e300])
def test_extreme_scales(scale):
    dz, s, rng, shape = problem((17, 16, 9), 2, FACES[0], 7)
    y, v = rng.standard_normal(shape), rng.standard_normal(shape)
    ref = wave.period(dz, y, v)
    got = [t / scale for t in s.wave_period(y * scale, v * scale)]
    close(got, ref)
    s.close()


def test_mixed_magnitudes_and_nonfinite():
    """Neighbours 200 binades apart, and infinities / NaN, end where the oracle has them."""
    dz, s, rng, shape = problem((20, 18), 2, FACES[0], 9)
    y = rng.standard_normal(shape) * 2.0 ** rng.integers(-200, 1, shape)
    v = np.zeros(shape)
    close([s.wave_period(y, v)[0]], [wave.period(dz, y, v)[0]])
    y = np.zeros(shape)
    y[9, 9] = np.nan
    assert dz.N > 9 + 11  # a node per step: the NaN has reached every corner
    assert torch.isnan(s.wave_period(y, v)[0]).all()
    s.close()
