"""Element rows times a vector (trace products and interior recovery) where the row counts are ragged against the
kernels' groups of eight rows, two groups per warp: random operators against NumPy in FP64."""
import math

import numpy as np
import pytest

from hdg_cases import Case, GpuCase

pytestmark = pytest.mark.gpu

CASES = [Case(f"euler2d_p{p}", 2, 2, p, 4.0, 0.5, 0.0, 0.71, "vortex", noise=0.0) for p in (1, 2, 3, 4)]
CASES += [Case(f"ns3d_p{p}", 3, 2, p, 2 * math.pi, 0.1, 1600.0, 0.71, "tgv", noise=0.0) for p in (1, 2)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: c.name)
def test_products_at_ragged_row_counts(case):
    from oracle.mesh import Mesh
    gc = GpuCase(case)
    torch, i = gc.torch, gc.info
    E, nv, nt = i["n_elem"], i["nv"], i["nt"]
    mesh = Mesh(case.dim, case.n, 0.0, case.L, case.p)
    rng = np.random.default_rng(nt)
    S = rng.normal(size=(E, nt, nt))
    rec = rng.normal(size=(E, nv * nt + nv))
    x = rng.normal(size=tuple(gc.Vhat.shape))
    xd, yd, dV = torch.from_numpy(x).to(gc.dev), torch.empty_like(gc.Vhat), torch.empty_like(gc.V)
    gc.S.copy_(torch.from_numpy(S))
    gc.recov.copy_(torch.from_numpy(rec))
    gc.hdg.hdg_trace_matvec(gc.ctx.handle, gc.S, xd, yd)
    gc.hdg.hdg_recover_interior(gc.ctx.handle, gc.recov, xd, dV)
    y, yabs = np.zeros_like(x), np.zeros_like(x)
    dV = dV.cpu().numpy().reshape(E, nv)
    for e in range(E):
        f, k = mesh.face_of[e][:, None], mesh.fnode_map[e]
        xe = x[f, k].ravel()
        X, y0 = rec[e, :nv * nt].reshape(nv, nt), rec[e, nv * nt:]
        # FP64 sums of nt products in another order: nt * 2^-53 of the sum of the magnitudes
        assert (np.abs(dV[e] - (-y0 - X @ xe)) <= 2.0 * (nt + 2) * 2.0 ** -53 * (np.abs(y0) + np.abs(X) @ np.abs(xe))).all()
        np.add.at(y, (f, k), (S[e] @ xe).reshape(*k.shape, -1))
        np.add.at(yabs, (f, k), (np.abs(S[e]) @ np.abs(xe)).reshape(*k.shape, -1))
    assert (np.abs(yd.cpu().numpy() - y) <= 2.0 * (nt + 2) * 2.0 ** -53 * yabs).all()
