"""On-chip step loops of several solvers at once, each in a thread and on a stream of its own: 2D and 3D
loops that fill the chip, cluster loops, FP64 ones and step-by-step solvers.  Each wait of such a loop
needs all of its blocks resident; a launch that got only some of them would run into its bound
(CMCG_ERR_DEVICE_TIMEOUT).  The results are those of each solver alone."""
import math
import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1903_12522_gb300 import cmcg  # noqa: E402

SOLVERS = [((700, 600), cmcg.FP32), ((128, 120, 110), cmcg.FP32), ((430, 300), cmcg.FP64), ((130, 90), cmcg.FP32),
           ((60, 50, 70), cmcg.FP64), ((96, 96, 90), cmcg.FP32)]


def make(n, precision):
    h = 1.0 / max(n)
    shape = tuple(m + 1 for m in reversed(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    faces = (cmcg.BC_ABC,) * (2 * len(n)) + (cmcg.BC_NEUMANN,) * (6 - 2 * len(n))
    c = 1 + 0.2 * torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)
    s = cmcg.Solver(n, h, c, 2 * math.pi / (12 * h), faces, precision=precision, dt=0.25 * h)
    y = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)
    return s, y


def test_threads():
    made = [make(*p) for p in SOLVERS]
    alone = [[*s.wave_period(y, y), *s.adjoint_period(y, y)] for s, y in made]
    torch.cuda.synchronize()
    errors = []

    def work(k):
        try:
            s, y = made[k]
            for _ in range(40):
                out = [*s.wave_period(y, y), *s.adjoint_period(y, y)]
                if not all(torch.equal(a, b) for a, b in zip(out, alone[k])):
                    errors.append((k, "differs"))
        except Exception as e:  # noqa: BLE001
            errors.append((k, repr(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(made))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for s, _ in made:
        s.close()
