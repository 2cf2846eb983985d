"""Rounding of the FP64 steps' integer stencil sums, against a period in extended precision.  A step
rounds three times (the sum, 2 y - y_prev, the fused update), each to nearest and independently of
the others, so that noise fields end within 3 sqrt(N) 2^-53 of the exact period; errors that all steps
share (a truncated sum, a rounded 4/3) grow with N instead and exceed it."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1903_12522_gb300 import cmcg  # noqa: E402

L = np.longdouble


def lap(y, order):
    out = np.zeros_like(y)
    for ax in range(y.ndim):
        n = y.shape[ax] - 1
        i = np.arange(n + 1)

        def at(k):
            j = np.abs(i + k)
            return np.take(y, np.where(j > n, 2 * n - j, j), axis=ax)

        if order == 2:
            out += 2 * y - at(1) - at(-1)
        else:
            out += L(5) / 2 * y - L(4) / 3 * (at(1) + at(-1)) + (at(2) + at(-2)) / L(12)
    return out


@pytest.mark.skipif(np.finfo(L).nmant < 60, reason="needs an extended long double")
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("n", [(30, 26, 24), (61, 40)])
def test_noise_period(n, order):
    h = 1.0 / max(n)
    shape = tuple(m + 1 for m in reversed(n))
    rng = np.random.Generator(np.random.PCG64(7))
    c = 1 + 0.5 * rng.random(shape)
    y, v = rng.standard_normal(shape), 50 * rng.standard_normal(shape)
    faces = (cmcg.BC_ABC,) * (2 * len(n)) + (cmcg.BC_NEUMANN,) * (6 - 2 * len(n))
    s = cmcg.Solver(n, h, c, 2 * math.pi / (12 * h), faces, precision=cmcg.FP64, order=order, dt=0.25 * h)
    N, dt = s.info["steps_per_period"], L(s.info["dt"])
    out = [x.cpu().numpy().reshape(shape) for x in s.wave_period(y, v)]
    s.close()
    kap = (c * c * s.info["dt"] ** 2 / (h * h)).astype(L)
    nb = sum(np.broadcast_to(np.isin(np.arange(m), (0, m - 1)).reshape([-1 if a == b else 1 for b in range(len(shape))]), shape)
             .astype(L) for a, m in enumerate(shape))
    beta = nb * np.sqrt(kap)
    y0, v = y.astype(L), v.astype(L)
    y1 = y0 + dt * (1 - beta) * v - kap * lap(y0, order) / 2
    for _ in range(N - 1):
        y0, y1 = y1, (2 * y1 - (1 - beta) * y0 - kap * lap(y1, order)) / (1 + beta)
    v = ((y1 - y0) / dt - kap * lap(y1, order) / (2 * dt)) / (1 + beta)
    for a, b in zip(out, (y1, v)):
        assert float(np.linalg.norm((a - b).astype(float).ravel()) / np.linalg.norm(b.astype(float).ravel())) <= 3 * math.sqrt(N) * 2.0**-53
