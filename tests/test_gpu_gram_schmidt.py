"""The Gram-Schmidt passes of a GMRES cycle with every number of basis vectors (1 to 30, groups of 8 and a remainder) and
vector lengths that are no multiple of a block: random operators that take more than one cycle."""
import pytest

from hdg_cases import Case, GpuCase

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p", [(2, 1), (3, 2), (9, 3)])   # 96, 324, 3888 unknowns
def test_cycles_over_all_basis_sizes(n, p):
    gc = GpuCase(Case("gs", 2, n, p, 4.0, 0.5, 0.0, 0.71, "vortex", noise=0.0))
    torch, hdg = gc.torch, gc.hdg
    nt = gc.info["nt"]
    gen = torch.Generator(device=gc.dev).manual_seed(3)
    gc.S.normal_(generator=gen)
    # 4 (p + 1) unknowns per face, four neighbour faces: the off-diagonal part has spectral radius sqrt(16 (p + 1)), so
    # that a residual of 1e-13 needs more than the 30 steps of one cycle
    gc.S += torch.eye(nt, dtype=torch.float64, device=gc.dev) * (0.8 * (16 * (p + 1)) ** 0.5)
    gc.g.normal_(generator=gen)
    x, r, b = (torch.empty_like(gc.Vhat) for _ in range(3))
    hdg.hdg_trace_matvec(gc.ctx.handle, torch.diag_embed(gc.g), torch.ones_like(b), b)
    it, res = hdg.hdg_trace_solve(gc.ctx.handle, gc.S, gc.g, x, hdg.HDG_SOLVER_GMRES, 1e-13, 3000)
    assert it > 30
    hdg.hdg_trace_matvec(gc.ctx.handle, gc.S, x, r)
    assert float((r + b).norm()) <= 1e-12 * float(b.norm())
