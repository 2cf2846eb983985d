"""2D step loops in one launch (bands of rows held on chip) against the CPU oracle: one band and many,
bands of the fewest rows, one to eight nodes per thread, the largest grid that fits and the first
that does not, loops longer than one launch, faces of every kind, sources on faces and inside.

Tolerances, relative to the largest value: FP64 as in test_gpu_step_soft (4 N^2 2^-53, N <= 47);
FP32 the same with 2^-24: 4 N^2 2^-24 <= 5.3e-4."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import wave  # noqa: E402
from oracle.grid import Discretization  # noqa: E402
from paper_1903_12522_gb300 import cmcg  # noqa: E402

TOL = {cmcg.FP64: 1e-12, cmcg.FP32: 5.3e-4}
SIZES = [(2, 2), (5, 2), (2, 300), (63, 64), (64, 63), (130, 40), (33, 200), (301, 9), (300, 303), (700, 6)]


def problem(n, order, faces, precision, ppw=10.0, dt_scale=1.0):
    if order == 4:
        faces = tuple(1 if f == 2 else f for f in faces)
    rng = np.random.Generator(np.random.PCG64(11))
    shape = tuple(m + 1 for m in reversed(n))
    h = 1.0 / max(n)
    c = rng.uniform(1.0, 2.0, shape)
    dt = dt_scale * (0.9 if order == 2 else 0.75) * h / (2.0 * np.sqrt(2.0))
    omega = 2 * np.pi / (ppw * h)
    dz = Discretization(n, h, c, omega, faces, dt, order=order)
    s = cmcg.Solver(n, h, c, omega, faces, order=order, dt=dt, precision=precision)
    return dz, s, rng, shape


def close(got, ref, tol):
    scale = max(np.abs(r).max() for r in ref)
    for a, b in zip(got, ref):
        assert np.abs(a.cpu().numpy() - b).max() <= tol * scale


@pytest.mark.parametrize("precision", [cmcg.FP64, cmcg.FP32])
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("n", SIZES)
def test_periods_match_oracle(n, order, precision):
    tol = TOL[precision]
    for faces in ((0,) * 6, (2, 0, 1, 0, 1, 1)):
        dz, s, rng, shape = problem(n, order, faces, precision)
        y, v = rng.standard_normal(shape), rng.standard_normal(shape) * dz.omega
        f = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
        for src in ((None, None), (f * dz.omega ** 2, None), (None, f)):
            F = None if src[0] is None and src[1] is None else dz.load(*src)
            for _ in range(2):  # a second period continues the bands' step counts
                got = s.wave_period(y, v, *src)
            ref = wave.period(dz, y, v, F)
            close([got[0], got[1] / dz.omega], [ref[0], ref[1] / dz.omega], tol)
        got = s.adjoint_period(y, v)
        close(got, wave.transposed_period(dz, y, v), tol)
        s.close()


@pytest.mark.parametrize("precision", [cmcg.FP64, cmcg.FP32])
def test_loop_longer_than_one_launch(precision):
    # 467 steps per period: three launches, the source factors of each its own
    dz, s, rng, shape = problem((70, 65), 2, (0,) * 6, precision, ppw=10.0, dt_scale=0.068)
    assert dz.N > 400
    y, v = rng.standard_normal(shape), np.zeros(shape)
    f = (rng.standard_normal(shape) + 0j) * dz.omega ** 2
    tol = 4 * dz.N ** 2 * (2.0 ** -53 if precision == cmcg.FP64 else 2.0 ** -24) / 10.0
    got = s.wave_period(y, v, f)
    ref = wave.period(dz, y, v, dz.load(f, None))
    close([got[0], got[1] / dz.omega], [ref[0], ref[1] / dz.omega], tol)
    close(s.adjoint_period(y, y), wave.transposed_period(dz, y, y), tol)
    s.close()


@pytest.mark.parametrize("n", [(1023, 1030), (1100, 1100), (783, 780), (800, 800)])
def test_largest_that_fits_and_first_that_does_not(n):
    # FP64 takes 512 threads of at most eight nodes on each SM, FP32 1024; past that the loop runs
    # step by step.  FP32 against FP64 on the GPU (the oracle's sparse matrix takes too long here).
    rng = np.random.Generator(np.random.PCG64(3))
    shape = tuple(m + 1 for m in reversed(n))
    h = 1.0 / max(n)
    c = rng.uniform(1.0, 2.0, shape)
    y, v = rng.standard_normal(shape), np.zeros(shape)
    out = {}
    for precision in (cmcg.FP64, cmcg.FP32):
        s = cmcg.Solver(n, h, c, 2 * np.pi / (10 * h), (0,) * 6, dt=0.9 * h / (2 * np.sqrt(2)), precision=precision)
        out[precision] = s.wave_period(y, v)[0], s.adjoint_period(y, y)[0]
        s.close()
    for a, b in zip(out[cmcg.FP32], out[cmcg.FP64]):
        assert (a - b).abs().max() <= TOL[cmcg.FP32] * b.abs().max()
