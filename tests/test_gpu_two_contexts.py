"""Two contexts of different sizes alive on one GPU: a kernel's dynamic shared-memory limit belongs to the kernel and
the device, so a call of the smaller context may not lower it under the larger one's."""
import math

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


class Flow:
    """A perturbed Taylor-Green state on 6 n^3 tetrahedra and the buffers of its linearisation."""

    def __init__(self, n, p, degrees=None):
        import torch
        from paper_1808_05066_gb300 import hdg
        self.hdg, self.torch = hdg, torch
        pe = None if degrees is None else np.resize(np.array(degrees, dtype=np.int8), 6 * n ** 3)
        self.mesh = hdg.Mesh(3, n, 0.0, 2 * math.pi, p, p_per_elem=pe)
        self.ctx = hdg.Context(self.mesh, 1.4, 0.1, 1600.0, 0.71)
        xn, xt, _ = self.mesh.coords()
        self.V, self.Vhat = self._entropy(xn), self._entropy(xt)
        self.Vhat = torch.from_numpy(wl.perturb(self.Vhat.cpu().numpy(), 1e-3, 5)).cuda().contiguous()
        i = self.mesh.info
        self.out = {k: torch.empty(i["len_" + k], dtype=torch.float64, device="cuda") for k in ("S", "g", "recov", "R")}
        self.status = torch.zeros(i["n_elem"], dtype=torch.int32, device="cuda")

    def _entropy(self, x):
        rho, vel, p = wl.tgv_field(x + 0.3, 0.1)
        prim = self.torch.from_numpy(np.concatenate([rho[..., None], vel, p[..., None]], -1)).cuda().contiguous()
        out = self.torch.empty_like(prim)
        self.hdg.hdg_prim_to_entropy(self.ctx.handle, prim, prim.numel() // 5, out)
        return out

    def assemble(self):
        o = self.out
        self.hdg.hdg_assemble_condense(self.ctx.handle, self.V, self.Vhat, None, 20.0, self.hdg.HDG_PREC_FP64, o["S"],
                                       o["g"], o["recov"], o["R"], self.status)
        self.torch.cuda.synchronize()
        assert int(self.status.abs().sum()) == 0
        return {k: v.clone() for k, v in o.items()}


def test_mixed_degree_assembly():
    large, small = Flow(1, 0, (4, 1, 3, 2, 4, 3)), Flow(1, 0, (1, 2, 2, 1, 1, 2))
    first = large.assemble()
    small.assemble()
    for k, v in large.assemble().items():
        assert large.torch.equal(v, first[k]), k


def _solve(flow):
    """GMRES into a new output buffer: a recorded cycle refers to its buffers and is recorded again."""
    x = flow.torch.empty_like(flow.Vhat)
    it, res = flow.hdg.hdg_trace_solve(flow.ctx.handle, flow.out["S"], flow.out["g"], x, flow.hdg.HDG_SOLVER_GMRES,
                                       1e-10, 600)
    assert it > 1 and res <= 1e-10
    return x


def test_trace_products():
    large, small = Flow(2, 3), Flow(2, 2)   # rings of 200 and 120 columns
    for f in (large, small):
        f.assemble()
    xs = [_solve(f) for f in (large, small, large)]
    torch = large.torch
    assert float(torch.linalg.norm(xs[2] - xs[0])) <= 1e-6 * float(torch.linalg.norm(xs[0]))
    c, r = large.hdg.hdg_ctx_trace_cycles(large.ctx.handle)
    assert c == r                           # every cycle a graph replay: nothing was refused while recording


def test_mixed_degree_preconditioner():
    large, small = Flow(2, 0, (4, 1, 3, 2, 4, 3)), Flow(2, 0, (1, 2, 2, 1, 1, 2))   # faces of 75 and 30 unknowns
    for f in (large, small):
        f.assemble()
    xs = [_solve(f) for f in (large, small, large)]
    torch = large.torch
    assert float(torch.linalg.norm(xs[2] - xs[0])) <= 1e-6 * float(torch.linalg.norm(xs[0]))
