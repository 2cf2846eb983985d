"""Engine slots whose step loops run in one launch each (2D grids that fit a cluster) beside slots that
stay in the batched kernel (3D, and 2D grids past a cluster), over grids of one band, of a cluster with
one to three chunks per thread, the largest that fits and the next one, and both orders: the same bits
alone, in the mix, and without graphs."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1903_12522_gb300 import cmcg  # noqa: E402

GRIDS = [((17, 9), 2), ((130, 61), 4), ((250, 255), 2), ((384, 330), 2), ((442, 442), 2), ((460, 460), 2), ((12, 14, 10), 2)]


def problem(n, order):
    h = 1.0 / max(n)
    shape = tuple(m + 1 for m in reversed(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    c = 1 + 0.3 * torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)
    f = torch.randn(shape, generator=gen, device="cuda", dtype=torch.complex128)
    faces = (cmcg.BC_ABC,) * (2 * len(n)) + (cmcg.BC_NEUMANN,) * (6 - 2 * len(n))
    return dict(n=n, h=h, c=c, omega=2 * math.pi / (12 * h), faces=faces), dict(order=order, dt=0.25 * h), f


def run(which, precision, flags, max_iter):
    engine = cmcg.Engine(len(which), flags=flags)
    problems = [problem(*GRIDS[i]) for i in which]
    torch.cuda.synchronize()
    solvers = [cmcg.Solver(**p, **o, precision=precision, flags=cmcg.FLAG_INEXACT_RIESZ, max_iter=max_iter,
                           stream=engine.stream) for p, o, _ in problems]
    slots = [engine.submit(s, f, None, tol=1e-9) for s, (_, _, f) in zip(solvers, problems)]
    done = []
    while len(done) < len(slots):
        done += engine.tick()
    out = [engine.result(s) for s in slots]
    torch.cuda.synchronize()
    engine.close()
    for s in solvers:
        s.close()
    return out


@pytest.mark.parametrize("precision", [cmcg.FP32, cmcg.MIXED])
def test_same_bits_alone_in_the_mix_and_without_graphs(precision):
    mix = run(range(len(GRIDS)), precision, 0, 5)
    plain = run(range(len(GRIDS)), precision, cmcg.ENGINE_NO_GRAPH, 5)
    for i, (w, st) in enumerate(mix):
        assert st["iterations"] == 5
        assert torch.equal(w, plain[i][0])
        assert torch.equal(w, run([i], precision, 0, 5)[0][0])
