"""The checked library (see test_gpu_checked) over the kernels that its other cases do not reach: steps on
padded rows where the on-chip loops do not take the grid, first-order rows, the V-cycle's coarse end in a
cluster (nested and ragged) and the small-grid PCG.  No out-of-range index, and the results are FP64's to
FP32 rounding (2e-5) or, for the Riesz map, those of the map without clusters to 1e-9."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1903_12522_gb300 import cmcg  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import math
import torch
from paper_1903_12522_gb300 import cmcg

assert cmcg.load()._name == cmcg.LIB_CHECKED_PATH


def clean(tag):
    code, count, site, index = cmcg.cmcg_check_status()
    assert code == cmcg.OK and count == 0, (tag, code, count, site, index)


def near(a, b, tol, tag):
    assert (a - b).norm() <= tol * b.norm(), tag


def solver(n, precision, order=2, faces=None, **kw):
    h = 1.0 / max(n)
    shape = tuple(m + 1 for m in reversed(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(2)
    c = 1 + torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)
    faces = faces or (cmcg.BC_ABC,) * (2 * len(n)) + (cmcg.BC_NEUMANN,) * (6 - 2 * len(n))
    s = cmcg.Solver(n, h, c, 2 * math.pi / (10 * h), faces, precision=precision, order=order, dt=0.2 * h, **kw)
    return s, lambda *k: torch.randn((*k, *shape), generator=gen, device="cuda", dtype=torch.float64)


for n, order in (((9, 7, 5), 4), ((31, 18, 9), 4), ((201, 150, 97), 2)):
    out = []
    for precision in (cmcg.FP64, cmcg.FP32):
        s, rnd = solver(n, precision, order)
        y, f = rnd(), torch.complex(rnd(), rnd()) * 1e3
        out.append([*s.wave_period(y, y, f), *s.wave_period(y, y, None, f), *s.adjoint_period(y, y)])
        s.close()
    clean(f"rows {n} {order}")
    for a, b in zip(out[1], out[0]):
        near(a, b, 2e-5, n)
for n in ((2, 2, 2), (9, 5, 4), (70, 33, 21)):
    out = []
    for precision in (cmcg.FP64, cmcg.FP32):
        s, rnd = solver(n, precision, flags=cmcg.FLAG_FIRST_ORDER)
        s0, y, f = rnd(4).reshape(-1), rnd(4).reshape(-1), (torch.complex(rnd(), rnd()) * max(n)).reshape(-1)
        out.append([s.fo_period(s0), s.fo_period(s0, f, f), s.fo_adjoint_period(y)])
        s.close()
    clean(f"first order {n}")
    for a, b in zip(out[1], out[0]):
        near(a, b, 2e-5, n)
for n in ((17, 20), (64, 64), (101, 86), (257, 300), (12, 9, 10), (33, 30, 29), (50, 47, 44)):
    s, rnd = solver(n, cmcg.FP64, faces=(cmcg.BC_DIRICHLET,) + (cmcg.BC_ABC,) * 5)
    rhs = rnd()
    x, code = s.riesz(rhs)
    assert code == cmcg.OK
    clean(f"riesz {n}")
    cmcg.cmcg_no_cluster_selftest(s.handle)
    near(x, s.riesz(rhs)[0], 1e-9, n)
    clean(f"riesz {n} without clusters")
    s.close()
print("CHECKED OK")
'''


def test_no_out_of_range_index():
    from paper_1903_12522_gb300 import build

    if not os.path.exists(cmcg.LIB_CHECKED_PATH):
        build.build(checked=True)
    env = dict(os.environ, CMCG_CHECKED="1", PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and "CHECKED OK" in r.stdout, r.stdout[-2000:] + r.stderr[-3000:]
