"""The mixed form's assembly on meshes of few tiles, whose columns several CTAs share, and of many, where a persistent CTA
goes from the rows with a viscous part to those without and the last chunk of elements is ragged."""
import math

import pytest

from hdg_cases import Case, GpuCase, rel_fro

pytestmark = pytest.mark.gpu


# chunks of these sizes deal the columns to 20, 10, 2 parts and one (3D, 20 test nodes), 15, 8, 2 and one (2D, 15), 6 and one (2D Euler, 6)
@pytest.mark.parametrize("case,chunks", [
    (Case("ns3d_p3", 3, 5, 3, 2 * math.pi, 0.1, 1600.0, 0.71, "tgv"), (6, 48, 300, 750)),
    (Case("ns2d_p4", 2, 24, 4, 30.0, 0.3, 1000.0, 0.71, "vortex"), (14, 128, 500, 1152)),
    (Case("euler2d_p2", 2, 24, 2, 30.0, 0.5, 0.0, 0.71, "vortex"), (9, 1152)),
], ids=lambda c: getattr(c, "name", None))
def test_parts_give_the_same_bits(case, chunks, monkeypatch):
    monkeypatch.setenv("HDG_COND_VARIANT", "2")   # one condensation for all
    ref = None
    for ch in chunks:
        monkeypatch.setenv("HDG_ELEMENT_CHUNK", str(ch))
        gc = GpuCase(case)
        gc.assemble(gc.history(), precision=1)
        assert int(gc.status.abs().sum()) == 0
        out = [t.clone() for t in (gc.S, gc.g, gc.recov, gc.R)]
        if ref is not None:
            for a, b in zip(out, ref):
                assert gc.torch.equal(a, b), ch
        ref = out


def test_many_tiles_and_a_ragged_chunk():
    gc = GpuCase(Case("ns3d_p1", 3, 12, 1, 2 * math.pi, 0.1, 1600.0, 0.71, "tgv"))   # 8,192 and 2,176 elements
    hist = gc.history()
    gc.assemble(hist, precision=0)
    ref = {k: getattr(gc, k).cpu().numpy().copy() for k in ("S", "g")}
    gc.assemble(hist, precision=1)
    assert int(gc.status.abs().sum()) == 0
    for k in ref:
        got = getattr(gc, k).cpu().numpy()
        assert max(rel_fro(got[e], ref[k][e]) for e in range(gc.info["n_elem"])) <= 1e-10, k
