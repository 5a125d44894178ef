"""The bounded waits of the streaming kernels, run out on purpose: a hook makes the host ask for a first operand copy that
is never issued, the kernel gives up after about a second a wait, drains its other copies, reports and returns. Nothing
faults, and the context stays usable."""
import time

import pytest

from hdg_cases import CASES, GpuCase

pytestmark = pytest.mark.gpu


def _code(fn):
    from paper_1808_05066_gb300 import hdg
    with pytest.raises(hdg.HdgError) as ei:
        fn()
    return ei.value.code


def test_mixed_assembly(monkeypatch):
    """18 triangles: the first CTA takes a part of the first tile of rows with a viscous part, elements 0 to 13. Exactly
    these carry TIMEOUT, and nothing else, when the recomputation is off; with it they are the FP64 form's bit for bit."""
    monkeypatch.setenv("HDG_ASM_STALL_FIRST_COPY", "1")
    monkeypatch.setenv("HDG_COND_VARIANT", "2")
    gc = GpuCase(CASES["ns2d_p3"])
    hdg, torch = gc.hdg, gc.torch
    hist = gc.history()
    outs = lambda: [t.clone() for t in (gc.S, gc.g, gc.recov, gc.R)]
    gc.assemble(hist, precision=0)
    fp64 = outs()
    gc.assemble(hist, precision=1)
    st = gc.status.cpu().numpy()
    assert (st[:14] == hdg.HDG_ELEM_FP64).all() and (st[14:] == 0).all()
    for x, y in zip(outs(), fp64):
        assert torch.equal(x[:14], y[:14])
    hdg.hdg_ctx_set_refinement(gc.ctx.handle, 1e-10, False)
    gc.assemble(hist, precision=1)
    st = gc.status.cpu().numpy()
    assert (st[:14] & hdg.HDG_ELEM_TIMEOUT).all() and not (st[:14] & hdg.HDG_ELEM_SINGULAR).any() and (st[14:] == 0).all()
    rest = outs()
    V, Vh = gc.V.clone(), gc.Vhat.clone()
    code = _code(lambda: hdg.hdg_newton_solve(gc.ctx.handle, V, Vh, hist, gc.case.mass_coef, 1, 1e-10, 2))
    assert code == hdg.HDG_ERR_TIMEOUT
    gc.assemble(hist, precision=0)                     # the context still works
    assert all(torch.equal(x, y) for x, y in zip(outs(), fp64)) and int(gc.status.abs().sum()) == 0
    monkeypatch.delenv("HDG_ASM_STALL_FIRST_COPY")     # and the other CTAs' elements were right
    free = GpuCase(CASES["ns2d_p3"])
    free.assemble(hist, precision=1)
    assert int(free.status.abs().sum()) == 0
    for x, y in zip(rest, (free.S, free.g, free.recov, free.R)):
        assert torch.equal(x[14:], y[14:])


def test_trace_product(monkeypatch):
    """The GMRES product of large elements (one iteration): HDG_ERR_TIMEOUT, and the next solve without the hook
    converges."""
    case = CASES["ns3d_p2"]
    monkeypatch.setenv("HDG_MATVEC_STALL_FIRST_COPY", "1")
    gc = GpuCase(case)
    hdg = gc.hdg
    gc.assemble(gc.history())
    x = gc.torch.empty_like(gc.Vhat)
    code = _code(lambda: hdg.hdg_trace_solve(gc.ctx.handle, gc.S, gc.g, x, hdg.HDG_SOLVER_GMRES, 1e-10, 1))
    assert code == hdg.HDG_ERR_TIMEOUT
    y = gc.torch.empty_like(gc.Vhat)
    hdg.hdg_trace_matvec(gc.ctx.handle, gc.S, gc.Vhat, y)   # the context still works
    assert bool(gc.torch.isfinite(y).all())
    monkeypatch.delenv("HDG_MATVEC_STALL_FIRST_COPY")
    free = GpuCase(case)
    it, res = hdg.hdg_trace_solve(free.ctx.handle, gc.S, gc.g, x, hdg.HDG_SOLVER_GMRES, 1e-10, 600)
    assert it > 1 and res <= 1e-10


@pytest.mark.parametrize("hook", ["HDG_ASM_STALL_FIRST_COPY", "HDG_MATVEC_STALL_FIRST_COPY"])
def test_waits_last_about_a_second(hook, monkeypatch):
    """Two waits in a row run out (the operand's and its drain's): two seconds, and three to launch and return."""
    monkeypatch.setenv("HDG_COND_VARIANT", "2")
    GpuCase(CASES["ns3d_p2"]).assemble(None, precision=1)   # kernels are loaded
    monkeypatch.setenv(hook, "1")
    gc = GpuCase(CASES["ns3d_p2"])
    hdg = gc.hdg
    gc.assemble(gc.history())
    x = gc.torch.empty_like(gc.Vhat)
    t = time.monotonic()
    if "ASM" in hook:
        gc.assemble(gc.history(), precision=1)
        assert (gc.status == hdg.HDG_ELEM_FP64).any()
    else:
        _code(lambda: hdg.hdg_trace_solve(gc.ctx.handle, gc.S, gc.g, x, hdg.HDG_SOLVER_GMRES, 1e-10, 1))
    assert 0.9 < time.monotonic() - t < 5.0
