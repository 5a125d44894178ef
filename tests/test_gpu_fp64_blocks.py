"""FP64 element blocks at the sizes where the contraction's 2 x 2 tiles and the condensation's column
and row blocks are ragged: odd node and face-node counts, interior sizes that are no multiple of the
triangular solve's block, fewer columns than a block. Against the oracle, element by element."""
import math

import numpy as np
import pytest

from hdg_cases import Case, GpuCase, oracle_hist, oracle_setup, rel_fro

pytestmark = pytest.mark.gpu

CASES = [Case(f"euler2d_p{p}", 2, 2, p, 4.0, 0.5, 0.0, 0.71, "vortex") for p in (1, 3, 4)]
CASES += [Case(f"ns2d_p{p}", 2, 2, p, 4.0, 0.5, 500.0, 0.71, "vortex") for p in (1, 2)]
CASES += [Case("ns3d_p2", 3, 1, 2, 2 * math.pi, 0.1, 1600.0, 0.71, "tgv")]


@pytest.mark.parametrize("case", CASES, ids=lambda c: c.name)
def test_ragged_blocks_match_oracle(case):
    prob, Q, V, Vh = oracle_setup(case)
    hist = oracle_hist(prob, V, case)
    gc = GpuCase(case)
    gc.assemble(gc.history())
    assert int(gc.status.abs().sum()) == 0
    i = gc.info
    S, g, rec, R = (t.cpu().numpy() for t in (gc.S, gc.g, gc.recov, gc.R))
    for e in range(i["n_elem"]):
        q = None if Q is None else Q[e]
        ref = prob.condense(e, q, V[e], prob.gather_trace(Vh, e), case.mass_coef, hist[e])
        nq = 0 if q is None else q.size
        nv, nt = i["nv"], i["nt"]
        assert rel_fro(S[e], ref["S"]) <= 1e-10
        assert rel_fro(g[e], ref["g"]) <= 1e-10
        assert rel_fro(rec[e, :nv * nt].reshape(nv, nt), ref["X"][nq:]) <= 1e-10
        assert rel_fro(rec[e, nv * nt:], ref["y"][nq:]) <= 1e-10
        scale = max(np.abs(ref["Rl"][nq:]).max(), np.abs(ref["Rt"]).max(), np.abs(hist[e]).max(), 1.0)
        assert np.abs(R[e, :nv] - ref["Rl"][nq:]).max() <= 1e-12 * scale
        assert np.abs(R[e, nv:] - ref["Rt"]).max() <= 1e-12 * scale


@pytest.mark.parametrize("p", [3, 4])
def test_elements_past_the_small_mesh_rule_match_oracle(p):
    """2D meshes of more than 304 elements take the blocked kernels, smaller ones those for small elements: both sides of
    the line give the oracle's blocks on sampled elements, at the same tolerance."""
    for n in (12, 13):                                    # 288 and 338 triangles
        case = Case(f"ns2d_p{p}", 2, n, p, 4.0, 0.5, 500.0, 0.71, "vortex")
        prob, Q, V, Vh = oracle_setup(case)
        gc = GpuCase(case)
        hist = gc.history()
        gc.assemble(hist)
        assert int(gc.status.abs().sum()) == 0
        i = gc.info
        S, g, rec = (t.cpu().numpy() for t in (gc.S, gc.g, gc.recov))
        for e in (0, 1, i["n_elem"] - 1):
            he = prob.history_weak(e, [V[e] * (1 + 1e-3)], [case.mass_coef])
            ref = prob.condense(e, Q[e], V[e], prob.gather_trace(Vh, e), case.mass_coef, he)
            nv, nt = i["nv"], i["nt"]
            assert rel_fro(S[e], ref["S"]) <= 1e-10
            assert rel_fro(g[e], ref["g"]) <= 1e-10
            assert rel_fro(rec[e, :nv * nt].reshape(nv, nt), ref["X"][Q[e].size:]) <= 1e-10


@pytest.mark.parametrize("reynolds,p,sizes", [(500.0, 3, (23, 24)), (500.0, 4, (8, 9)), (0.0, 4, (12, 13))])
def test_both_sides_of_the_small_mesh_lines_match_oracle(reynolds, p, sizes):
    """The lines lie at seven, one and two elements per SM (1,064, 152 and 304 on 152 SMs)."""
    for n in sizes:
        case = Case(f"2d_p{p}", 2, n, p, 1.25 * n, 0.5, reynolds, 0.71, "vortex")
        prob, Q, V, Vh = oracle_setup(case)
        gc = GpuCase(case)
        gc.assemble(gc.history())
        assert int(gc.status.abs().sum()) == 0
        nv, nt = gc.info["nv"], gc.info["nt"]
        for e in (0, 1, gc.info["n_elem"] - 1):
            q = None if Q is None else Q[e]
            nq = 0 if q is None else q.size
            he = prob.history_weak(e, [V[e] * (1 + 1e-3)], [case.mass_coef])
            ref = prob.condense(e, q, V[e], prob.gather_trace(Vh, e), case.mass_coef, he)
            assert rel_fro(gc.S[e].cpu().numpy(), ref["S"]) <= 1e-10
            assert rel_fro(gc.g[e].cpu().numpy(), ref["g"]) <= 1e-10
            X = gc.recov[e, :nv * nt].cpu().numpy().reshape(nv, nt)
            assert rel_fro(X, ref["X"][nq:]) <= 1e-10
