"""The mixed form on point tensors beyond the float range (2^128 = 3.4e38), from an enormous time coefficient: its scales
are floats, so a row of such tensors may not come out finite. Every block is either flagged or the FP64 form's."""
import pytest

from hdg_cases import CASES, GpuCase, rel_fro

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mass_coef", [1e40, 1e45, 1e120, 1e250])
def test_flagged_or_exact(mass_coef):
    gc = GpuCase(CASES["ns2d_p3"])
    hdg, torch = gc.hdg, gc.torch
    hist = torch.empty_like(gc.V)
    hdg.hdg_history(gc.ctx.handle, gc.V, None, mass_coef, 0.0, hist)   # u^n = u: the residual stays small

    def assemble(precision):
        gc.status.zero_()
        hdg.hdg_assemble_condense(gc.ctx.handle, gc.V, gc.Vhat, hist, mass_coef, precision, gc.S, gc.g, gc.recov, gc.R,
                                  gc.status)
        torch.cuda.synchronize()
        nv, nt = gc.info["nv"], gc.info["nt"]
        return {"S": gc.S.cpu().numpy().copy(), "X": gc.recov[:, :nv * nt].cpu().numpy().copy()}, gc.status.cpu().numpy()

    ref, st = assemble(0)
    assert not st.any()
    hdg.hdg_ctx_set_refinement(gc.ctx.handle, 1e-10, False)   # no recomputation: the blocks of the mixed form itself
    got, st = assemble(1)
    for e in range(gc.info["n_elem"]):
        for k in ref:
            assert st[e] or rel_fro(got[k][e], ref[k][e]) <= 1e-10, (e, k)
