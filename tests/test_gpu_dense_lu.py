"""Blocked dense LU of the trace matrix at sizes that are ragged against its panels (8 columns), blocks (32) and tiles
(64) and against its clusters of eight blocks: random element operators, which need row interchanges throughout."""
import numpy as np
import pytest

from hdg_cases import Case, GpuCase

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p", [(2, 1), (2, 2), (3, 2), (5, 3), (12, 1)])   # 96, 144, 324, 1200, 3456 unknowns
def test_dense_solve_of_random_operators(n, p):
    gc = GpuCase(Case("lu", 2, n, p, 4.0, 0.5, 0.0, 0.71, "vortex", noise=0.0))
    torch, hdg = gc.torch, gc.hdg
    gen = torch.Generator(device=gc.dev).manual_seed(n + 10 * p)
    gc.S.normal_(generator=gen)
    gc.g.normal_(generator=gen)
    x, r, scale = torch.empty_like(gc.Vhat), torch.empty_like(gc.Vhat), torch.empty_like(gc.Vhat)
    b = torch.empty_like(gc.Vhat)
    hdg.hdg_trace_matvec(gc.ctx.handle, torch.diag_embed(gc.g), torch.ones_like(b), b)   # the assembled g
    for _ in range(2):                                   # the second solve replays the recorded factorisation
        hdg.hdg_trace_solve(gc.ctx.handle, gc.S, gc.g, x, hdg.HDG_SOLVER_DENSE, 1e-12, 1)
        hdg.hdg_trace_matvec(gc.ctx.handle, gc.S, x, r)  # K x = -g
        hdg.hdg_trace_matvec(gc.ctx.handle, gc.S.abs(), x.abs(), scale)
        # backward error of partial pivoting: 2^-53 times a growth of about n^(2/3) (231) times a few sqrt(n)
        assert float((r + b).abs().max()) <= 1e-11 * float(scale.max())
        gc.g.neg_()
        b.neg_()
    gc.S.zero_()
    with pytest.raises(hdg.HdgError) as ei:
        hdg.hdg_trace_solve(gc.ctx.handle, gc.S, gc.g, x, hdg.HDG_SOLVER_DENSE, 1e-12, 1)
    assert ei.value.code == hdg.HDG_ERR_SINGULAR
