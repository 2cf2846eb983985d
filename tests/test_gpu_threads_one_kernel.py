"""Threads whose launches take one kernel with different amounts of shared memory: Riesz maps on grids whose
V-cycles end in clusters of different sizes.  The limit that a launch needs is set for the kernel as a whole,
so one thread must not lower it between another's setting and launch.  The results are those of each alone."""
import math
import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1903_12522_gb300 import cmcg  # noqa: E402


def test_riesz_maps_of_different_grids():
    made = []
    for n in ((256, 256), (64, 64, 64), (300, 200), (100, 90, 80)):
        h = 1.0 / max(n)
        shape = tuple(m + 1 for m in reversed(n))
        gen = torch.Generator(device="cuda")
        gen.manual_seed(4)
        c = torch.ones(shape, device="cuda", dtype=torch.float64)
        faces = (cmcg.BC_ABC,) * (2 * len(n)) + (cmcg.BC_NEUMANN,) * (6 - 2 * len(n))
        s = cmcg.Solver(n, h, c, 2 * math.pi / (10 * h), faces, dt=0.4 * h)
        rhs = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)
        made.append((s, rhs - rhs.mean(), None))
    made = [(s, rhs, s.riesz(rhs)[0]) for s, rhs, _ in made]
    errors = []

    def work(k):
        s, rhs, alone = made[k]
        for _ in range(150):
            try:
                x, code = s.riesz(rhs)
                if code != cmcg.OK or not torch.equal(x, alone):
                    errors.append((k, code))
            except Exception as e:  # noqa: BLE001
                errors.append((k, repr(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(made))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]
    for s, _, _ in made:
        s.close()
