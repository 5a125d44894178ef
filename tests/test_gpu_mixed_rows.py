"""The mixed form's assembly product at the sizes where its 128-row tiles are ragged (fewer elements than
a tile, one more than a whole number of tiles) and on a field whose far part is exactly uniform, so
that whole operand rows are subnormal or zero: the mixed blocks against the FP64 form's, S and g within
the mixed form's 1e-10, no element flagged."""
import math

import pytest

from hdg_cases import Case, GpuCase, rel_fro

pytestmark = pytest.mark.gpu

CASES = [
    Case("ns3d_p3_6", 3, 1, 3, 2 * math.pi, 0.1, 1600.0, 0.71, "tgv"),          # 6 elements of 8 in a tile
    Case("ns3d_p1_162", 3, 3, 1, 2 * math.pi, 0.1, 1600.0, 0.71, "tgv"),        # 20 tiles and 2 elements
    Case("ns2d_p4_98", 2, 7, 4, 8.75, 0.3, 1000.0, 0.71, "vortex"),             # 7 tiles of 14 elements
    Case("ns2d_p4_128", 2, 8, 4, 10.0, 0.3, 1000.0, 0.71, "vortex"),            # 9 tiles and 2 elements
    Case("euler2d_p2_18", 2, 3, 2, 3.75, 0.5, 0.0, 0.71, "vortex"),             # value operators only, 8 a tile
    Case("ns2d_p3_far", 2, 24, 3, 30.0, 0.5, 5000.0, 0.71, "vortex", noise=0.0),  # e^{1 - r^2} underflows
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: c.name)
def test_ragged_tiles_and_uniform_far_field(case):
    gc = GpuCase(case)
    hist = gc.history()
    gc.assemble(hist, precision=0)
    ref = {k: getattr(gc, k).cpu().numpy().copy() for k in ("S", "g", "R")}
    gc.assemble(hist, precision=1)
    assert int(gc.status.abs().sum()) == 0
    S, g, R = (getattr(gc, k).cpu().numpy() for k in ("S", "g", "R"))
    for e in range(gc.info["n_elem"]):
        assert rel_fro(S[e], ref["S"][e]) <= 1e-10, e
        assert rel_fro(g[e], ref["g"][e]) <= 1e-10, e
    # the two forms' residuals may come from different kernels (small elements): FP64 rounding of the summed terms
    scale = max(abs(ref["R"]).max(), float(hist.abs().max()), 1.0)
    assert abs(R - ref["R"]).max() <= 1e-12 * scale
