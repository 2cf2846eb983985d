"""The bounded waits of step loops in one launch: with a limit of one poll a loop over several bands or
blocks gives up, the call returns CMCG_ERR_DEVICE_TIMEOUT, and the same handle, with its default limit again,
gives the bits that it gave before.  (No word is held back: a wait of one poll runs out by itself.)  In
periods of each kind of loop, in whole solves where the loop is in the run-up, the CG iterations or J, and in
the engine, whose other slots go on."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1903_12522_gb300 import cmcg  # noqa: E402


def make(n, precision, order=2, **kw):
    h = 1.0 / max(n)
    shape = tuple(m + 1 for m in reversed(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(6)
    faces = (cmcg.BC_ABC,) * (2 * len(n)) + (cmcg.BC_NEUMANN,) * (6 - 2 * len(n))
    c = 1 + 0.2 * torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)
    s = cmcg.Solver(n, h, c, 2 * math.pi / (12 * h), faces, precision=precision, order=order, dt=0.25 * h, **kw)
    y = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)
    return s, y, torch.complex(y, 0.5 * y) / h ** 2


def times_out(call):
    with pytest.raises(cmcg.CMCGError) as e:
        call()
    assert e.value.code == cmcg.ERR_DEVICE_TIMEOUT


# bands in a cluster, bands through L2, FP64, 4th order, 3D blocks
@pytest.mark.parametrize("n,precision,order", [((300, 303), cmcg.FP32, 2), ((1000, 900), cmcg.FP32, 2), ((430, 300), cmcg.FP64, 2),
                                               ((400, 300), cmcg.FP32, 4), ((96, 90, 80), cmcg.FP32, 2)])
def test_periods(n, precision, order):
    s, y, f = make(n, precision, order)

    def calls():
        return [*s.wave_period(y, y), *s.wave_period(y, y, f), *s.adjoint_period(y, y)]

    before = calls()
    for _ in range(2):
        cmcg.cmcg_loop_wait_selftest(s.handle, 1)
        for call in (lambda: s.wave_period(y, y), lambda: s.wave_period(y, y, f), lambda: s.adjoint_period(y, y)):
            times_out(call)
        cmcg.cmcg_loop_wait_selftest(s.handle, 0)
        assert all(torch.equal(a, b) for a, b in zip(before, calls()))
    s.close()


@pytest.mark.parametrize("kw", [dict(precision=cmcg.FP64), dict(precision=cmcg.FP32, flags=cmcg.FLAG_INEXACT_RIESZ),
                                dict(precision=cmcg.MIXED, flags=cmcg.FLAG_INEXACT_RIESZ, runup_periods=2),
                                dict(precision=cmcg.FP32, flags=cmcg.FLAG_NO_CG, runup_periods=3),
                                dict(precision=cmcg.FP32, flags=cmcg.FLAG_NO_CG | cmcg.FLAG_FILTER, runup_periods=3)])
def test_solves(kw):
    s, y, f = make((430, 300), max_iter=3, **kw)
    before = s.solve(f, tol=1e-12)[0]
    cmcg.cmcg_loop_wait_selftest(s.handle, 1)
    times_out(lambda: s.solve(f, tol=1e-12))
    # without statistics there is no J whose read would bring the status
    f_flat, u = f.reshape(-1), torch.empty_like(f).reshape(-1)
    torch.cuda.synchronize()
    assert cmcg.load().cmcg_solve(s.handle, f_flat.data_ptr(), None, 1e-12, u.data_ptr(), None) == cmcg.ERR_DEVICE_TIMEOUT
    cmcg.cmcg_loop_wait_selftest(s.handle, 0)
    assert torch.equal(before, s.solve(f, tol=1e-12)[0])
    s.close()


def test_engine_slot():
    results = []
    for limited in (False, True):
        engine = cmcg.Engine(2)
        made = [make(n, cmcg.FP32, flags=cmcg.FLAG_INEXACT_RIESZ, max_iter=4, stream=engine.stream) for n in ((300, 303), (260, 200))]
        torch.cuda.synchronize()
        slots = [engine.submit(s, f, None, tol=1e-12) for s, _, f in made]
        if limited:
            cmcg.cmcg_loop_wait_selftest(made[0][0].handle, 1)
        late = 0
        while engine.active():
            try:
                engine.tick()
            except cmcg.CMCGError as e:
                assert e.code == cmcg.ERR_DEVICE_TIMEOUT
                late += 1
        out = [engine.result(q) for q in slots]
        assert late == (1 if limited else 0)
        assert out[0][1]["status"] == (cmcg.ERR_DEVICE_TIMEOUT if limited else cmcg.NOT_CONVERGED)
        results.append(out[1])
        torch.cuda.synchronize()
        engine.close()
        for s, _, _ in made:
            s.close()
    assert results[0][1]["status"] == results[1][1]["status"] and torch.equal(results[0][0], results[1][0])
