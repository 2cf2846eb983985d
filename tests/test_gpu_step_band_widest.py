"""FP32 grids of three rows about the widest that one CTA holds (two float4 chunks per thread) and past
it, where the loop runs step by step, against the oracle; tolerance as in test_gpu_step_band."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import wave  # noqa: E402
from paper_1903_12522_gb300 import cmcg  # noqa: E402
from test_gpu_step_band import TOL, close, problem  # noqa: E402


@pytest.mark.parametrize("nx", [2723, 2727, 2728, 2730, 2891, 2892])
def test_three_rows(nx):
    for faces in ((0,) * 6, (2, 0, 0, 0, 1, 1)):
        dz, s, rng, shape = problem((nx, 2), 2, faces, cmcg.FP32)
        y, v = rng.standard_normal(shape), rng.standard_normal(shape) * dz.omega
        f = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
        for src in ((None, None), (f * dz.omega ** 2, None), (None, f)):
            F = None if src[0] is None and src[1] is None else dz.load(*src)
            got, ref = s.wave_period(y, v, *src), wave.period(dz, y, v, F)
            close([got[0], got[1] / dz.omega], [ref[0], ref[1] / dz.omega], TOL[cmcg.FP32])
        close(s.adjoint_period(y, v), wave.transposed_period(dz, y, v), TOL[cmcg.FP32])
        s.close()
