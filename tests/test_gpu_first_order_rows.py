"""First-order periods at the sizes where the padded FP32 rows and the split of the z-planes can go
wrong: rows of every remainder and the shortest ones, one plane per thread and two, mixed faces with
Dirichlet nodes, and sources everywhere, in single columns and on the faces only.  Against the oracle,
element by element; tolerances as for the other first-order periods (FP64 1e-12, FP32 2e-5 relative
L2)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import first_order as ofo  # noqa: E402
from oracle.grid import Discretization  # noqa: E402
from paper_1903_12522_gb300 import cmcg  # noqa: E402
from paper_1903_12522_gb300 import workloads as wl  # noqa: E402
from test_gpu_first_order import pack, rand_state, rel, solver_of  # noqa: E402

ABC, NEU, DIR = wl.ABC, wl.NEUMANN, wl.DIRICHLET
SIZES = [(2, 2, 2), (3, 4, 2), (4, 3, 5), (5, 7, 3), (6, 2, 9), (7, 5, 4), (33, 6, 5), (130, 9, 4), (6, 70, 40), (62, 61, 60)]
FACES = [(ABC,) * 6, (NEU, ABC, ABC, NEU, DIR, ABC)]


@pytest.mark.parametrize("faces", FACES)
@pytest.mark.parametrize("n", SIZES)
def test_periods(n, faces):
    h = 1.0 / max(n)
    shape = tuple(m + 1 for m in reversed(n))
    rng = np.random.Generator(np.random.PCG64(31))
    c = 1.0 + 0.6 * rng.random(shape)

    def cplx():
        return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex128) / h

    few = np.where(rng.random(shape) < 0.02, cplx(), 0)
    w = wl.Workload(name="rows", n=n, h=h, c=c, omega=2 * np.pi / (9 * h), faces=faces, dt_target=0.3 * h / 1.6)
    dz = Discretization(w.n, w.h, w.c, w.omega, w.faces, w.dt_target)
    st = ofo.Staggered(dz)
    for precision, tol in ((cmcg.FP64, 1e-12), (cmcg.FP32, 2e-5)):
        s = solver_of(w, precision)
        p0, v0 = rand_state(st, dz, 3)
        for f, g in ((None, None), (cplx(), None), (few, None), (None, cplx()), (few, cplx())):
            ref = pack(*st.period(p0, v0, dz.load(f, g) if f is not None or g is not None else None))
            assert rel(s.fo_period(pack(p0, v0), f, g).cpu().numpy(), ref) <= tol
        y = rand_state(st, dz, 4)
        assert rel(s.fo_adjoint_period(pack(*y)).cpu().numpy(), pack(*st.transposed_period(*y))) <= tol
        s.close()
