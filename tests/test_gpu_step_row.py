"""FP32 3D steps on padded rows against the flat z-pair kernels: the same bits, for every step variant
(forced from inside and from the faces, homogeneous, the adjoint's first and last), both orders,
mixed faces, an obstacle, rows of every remainder, the narrowest rows that take them and one
narrower, and loops of one and two steps."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1903_12522_gb300 import cmcg  # noqa: E402

SIZES = [(7, 3, 3), (8, 2, 2), (9, 5, 7), (10, 33, 4), (31, 30, 29), (32, 16, 17), (63, 40, 9), (130, 21, 12)]
FACES = [(0,) * 6, (1, 0, 0, 1, 2, 0)]


def periods(n, order, faces, tile, f, g, mask=None, steps=None):
    h = 1.0 / max(n)
    shape = tuple(m + 1 for m in reversed(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)

    def rnd():
        return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)

    c = 1 + torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)
    y, v = rnd(), 50 * rnd()
    amp = 1e3 * torch.complex(rnd(), rnd())
    omega = 2 * math.pi / (10 * h) if steps is None else 2 * math.pi / (steps * 0.2 * h)
    dt = (0.22 if order == 2 else 0.2) * h
    s = cmcg.Solver(n, h, c, omega, faces, mask=mask, precision=cmcg.FP32, order=order, tile=tile, dt=dt)
    if steps is not None:
        assert s.info["steps_per_period"] <= steps
    out = [*s.wave_period(y, v, amp if f else None, amp if g else None), *s.adjoint_period(y, v)]
    s.close()
    return out


@pytest.mark.parametrize("faces", FACES)
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("n", SIZES)
def test_same_bits_as_flat_kernels(n, order, faces):
    if order == 4:
        faces = tuple(1 if f == 2 else f for f in faces)
    mask = None
    if order == 2:
        mask = torch.zeros(tuple(m + 1 for m in reversed(n)), dtype=torch.uint8, device="cuda")
        mask[tuple(slice((m + 1) // 3, (m + 1) // 2 + 1) for m in reversed(n))] = 1
    for f, g, mk in ((0, 0, mask), (1, 0, None), (0, 1, mask), (1, 1, None)):
        a = periods(n, order, faces, (16, 0, 0, 3), f, g, mk)
        b = periods(n, order, faces, (0, 0, 0, 0), f, g, mk)
        for x, y in zip(a, b):
            assert torch.equal(x, y)


@pytest.mark.parametrize("steps", [2, 3])
def test_loops_of_one_and_two_steps(steps):
    a = periods((17, 9, 12), 2, (0,) * 6, (16, 0, 0, 3), 1, 1, steps=steps)
    b = periods((17, 9, 12), 2, (0,) * 6, (0, 0, 0, 0), 1, 1, steps=steps)
    for x, y in zip(a, b):
        assert torch.equal(x, y)


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("n", [(33, 30, 29), (9, 5, 7), (130, 21, 12), (301, 90, 101)])
def test_sources_at_a_few_nodes(n, order):
    # corners, the last planes, single nodes inside, and values that are zero in FP32
    shape = tuple(m + 1 for m in reversed(n))
    f = torch.zeros(shape, dtype=torch.complex128, device="cuda")
    for z, y, x in ((0, 0, 0), (-1, -1, -1), (n[2] // 2, 1, n[0] // 2), (n[2] - 1, n[1] // 2, 3), (3, 2, n[0] - 1), (4, n[1], 4)):
        f[z, y, x] = 3e3 - 2e3j
    f[f == 0] = 1e-60
    h = 1.0 / max(n)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    y = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)
    out = []
    for tile in ((16, 0, 0, 3), (0, 0, 0, 0)):
        s = cmcg.Solver(n, h, torch.ones_like(y), 2 * math.pi / (10 * h), (0,) * 6, precision=cmcg.FP32, order=order, tile=tile,
                        dt=0.3 * h)
        out.append([*s.wave_period(y, y, f, f), *s.wave_period(y, y, None, None), *s.wave_period(y, y, f, None)])
        s.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
