"""Dense trace solve with pivots whose reciprocal is no usable number: an infinite one gives that unknown the value zero
and leaves the others alone, a last one of 1e-310 divides, as in x / d."""
import pytest

from hdg_cases import Case, GpuCase

pytestmark = pytest.mark.gpu


def test_infinite_and_subnormal_pivots():
    gc = GpuCase(Case("lu", 2, 2, 1, 4.0, 0.5, 0.0, 0.71, "vortex", noise=0.0))   # 96 unknowns
    torch, hdg = gc.torch, gc.hdg
    # element operators that assemble to a diagonal matrix, and its diagonal
    d = torch.linspace(1.0, 2.0, gc.Vhat.numel(), dtype=torch.float64, device=gc.dev)
    d[7], d[40], d[-1] = float("inf"), float("inf"), 1e-310
    own = torch.full((gc.info["n_elem"],), 0.5, dtype=torch.float64, device=gc.dev)   # a face has two elements
    idx = torch.empty_like(gc.Vhat)
    # local number -> global unknown, from products with unit diagonals of single elements
    ids = torch.arange(1, d.numel() + 1, dtype=torch.float64, device=gc.dev).reshape(gc.Vhat.shape)
    nt = gc.info["nt"]
    tmap = torch.empty((gc.info["n_elem"], nt), dtype=torch.int64, device=gc.dev)
    for e in range(gc.info["n_elem"]):
        for r in range(nt):
            S = torch.zeros_like(gc.S)
            S[e, r, r] = 1.0
            hdg.hdg_trace_matvec(gc.ctx.handle, S, ids, idx)
            tmap[e, r] = int(idx.max()) - 1
    half = d[tmap] * own[:, None]
    gc.S.copy_(torch.diag_embed(half))
    b = torch.ones_like(d)
    b[-1] = 1e-310
    gc.g.copy_(-0.5 * b[tmap])                      # K x = -g
    x = torch.empty_like(gc.Vhat)
    hdg.hdg_trace_solve(gc.ctx.handle, gc.S, gc.g, x, hdg.HDG_SOLVER_DENSE, 1e-12, 1)
    assert float((x.flatten() - b / d).abs().max()) <= 1e-15
