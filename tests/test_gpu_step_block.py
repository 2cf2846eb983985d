"""FP32 3D 7-point step loops in one launch, the grid on chip, against the flat z-pair kernels: the
same bits, for every step variant (forced from inside and from the faces, homogeneous, the adjoint's
first and last), mixed faces, an obstacle, rows of every remainder, the narrowest rows that take it
and one narrower, one block, blocks along one axis, uneven blocks, the largest grids, loops of one
and two steps and of more steps than a launch holds; and, just past the largest, the padded-row
kernels that the same call goes to."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1903_12522_gb300 import cmcg  # noqa: E402

FLAT = (16, 0, 0, 3)
SIZES = [(3, 9, 9), (4, 3, 3), (5, 2, 2), (6, 2, 30), (7, 40, 2), (9, 5, 7), (31, 30, 29), (64, 65, 66), (100, 200, 31),
         (122, 96, 149), (128, 128, 128), (399, 60, 50)]
PAST = [(4997, 3, 3), (4998, 5, 2), (4999, 2, 4), (5000, 3, 3)]
FACES = [(0,) * 6, (1, 0, 0, 1, 2, 0)]


def periods(n, faces, tile, f, g, mask=None, steps=None, repeat=1):
    h = 1.0 / max(n)
    shape = tuple(m + 1 for m in reversed(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)

    def rnd():
        return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)

    c = 1 + torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)
    y, v = rnd(), 50 * rnd()
    amp = 1e3 * torch.complex(rnd(), rnd())
    omega = 2 * math.pi / ((10 if steps is None else 0.2 * steps) * h)
    s = cmcg.Solver(n, h, c, omega, faces, mask=mask, precision=cmcg.FP32, tile=tile, dt=0.22 * h)
    out = []
    for _ in range(repeat):
        out += [*s.wave_period(y, v, amp if f else None, amp if g else None), *s.adjoint_period(y, v)]
    out.append(torch.tensor(float(s.info["steps_per_period"])))
    s.close()
    return out


def compare(n, faces, f, g, mask=None, **kw):
    a = periods(n, faces, FLAT, f, g, mask, **kw)
    b = periods(n, faces, (0, 0, 0, 0), f, g, mask, **kw)
    for x, y in zip(a, b):
        assert torch.isfinite(x).all() and torch.equal(x, y)
    return int(a[-1])


@pytest.mark.parametrize("faces", FACES)
@pytest.mark.parametrize("n", SIZES + PAST)
def test_same_bits_as_flat_kernels(n, faces):
    mask = torch.zeros(tuple(m + 1 for m in reversed(n)), dtype=torch.uint8, device="cuda")
    mask[tuple(slice((m + 1) // 3, (m + 1) // 2 + 1) for m in reversed(n))] = 1
    for f, g, mk in ((0, 0, mask), (1, 0, None), (0, 1, mask), (1, 1, None)):
        compare(n, faces, f, g, mk)


@pytest.mark.parametrize("steps", [2, 3])
def test_loops_of_one_and_two_steps(steps):
    assert compare((17, 9, 12), (0,) * 6, 1, 1, steps=steps, repeat=2) <= steps


def test_more_steps_than_a_launch_holds():
    assert compare((33, 21, 12), (0,) * 6, 0, 1, steps=450, repeat=2) > 401
