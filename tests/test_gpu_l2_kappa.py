"""CMCG_FLAG_L2_KAPPA raises the process's persisting-L2 set-aside to the size of the kappa that the step
kernels read: the padded copy, the flat one with another step scheme, and none where the step loops hold
the grid on chip and read kappa once."""
import ctypes
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1903_12522_gb300 import cmcg  # noqa: E402

LIMIT_PERSISTING = 6  # cudaLimitPersistingL2CacheSize


def set_aside():
    rt = ctypes.CDLL("libcudart.so.13")
    v = ctypes.c_size_t()
    assert rt.cudaDeviceGetLimit(ctypes.byref(v), LIMIT_PERSISTING) == 0
    return v.value


@pytest.mark.parametrize("n,order,tile,pitch", [((96, 90, 80), 2, (0, 0, 0, 0), None), ((96, 90, 80), 2, (16, 0, 0, 3), 97),
                                                ((201, 150, 160), 2, (0, 0, 0, 0), 204), ((201, 150, 160), 2, (16, 0, 0, 3), 202),
                                                ((97, 90, 80), 4, (0, 0, 0, 0), 100), ((600, 500), 2, (0, 0, 0, 0), None),
                                                ((1500, 1400), 2, (0, 0, 0, 0), 1501)])
def test_set_aside(n, order, tile, pitch):
    torch.cuda.synchronize()
    before = set_aside()
    h = 1.0 / max(n)
    shape = tuple(m + 1 for m in reversed(n))
    c = torch.ones(shape, device="cuda", dtype=torch.float64)
    torch.cuda.synchronize()
    s = cmcg.Solver(n, h, c, 2 * math.pi / (10 * h), (0,) * 6, precision=cmcg.FP32, order=order, tile=tile, dt=0.25 * h,
                    flags=cmcg.FLAG_L2_KAPPA, stream=torch.cuda.Stream())
    want = 0 if pitch is None else 4 * pitch * math.prod(shape[:-1])
    during = set_aside()
    s.close()
    # (the device rounds a limit up)
    assert during == before if want == 0 else during >= max(want, before) and (before >= want or during <= want + (8 << 20))
    assert set_aside() == before
