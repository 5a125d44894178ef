"""The work counts behind the reported fractions, against enumerations of the contraction's terms and the kernels' own sizes."""
import pytest

from paper_1808_05066_gb300 import workload as w

NS3 = dict(dim=3, m=5, Np=20, Nf=10, nF=4, NG=64, NGF=16, nv=100, nt=200)     # tetrahedra, p = 3
EU2 = dict(dim=2, m=4, Np=6, Nf=3, nF=3, NG=9, NGF=3, nv=24, nt=36)           # triangles, p = 2


def _contraction(i, viscous):
    """Multiply-adds term by term: one per point, test function or row, and trial column with an entry."""
    D, M, NP, NF, NFN, NG, NGF = i["dim"], i["m"], i["Np"], i["nF"], i["Nf"], i["NG"], i["NGF"]
    n = 0
    for a in range(M):
        for b in range(M):
            visc = viscous and a > 0 and b > 0
            for f in range(NF):
                cols = [(None, 1 + (D if visc else 0))] * NP                 # trial column: terms at a face point
                cols += [(g, (g == f) + visc) for g in range(NF) for _ in range(NFN)]
                n += NGF * sum(t for _, t in cols) + NFN * NGF * sum(1 for _, t in cols if t)
            n += NP * NG * (1 + D) + NP * NP * NG                            # value operator: left factor, product
            if visc:
                for o in range(D + 1):                                       # gradient operators
                    n += NP * NG * D + (NP * NP * NG if o < D else 0) + NP * NFN * NG
    return n


@pytest.mark.parametrize("info,viscous", [(NS3, True), (EU2, False)])
def test_contraction_count(info, viscous):
    assert w.flops_per_element(info, viscous, "assemble") == 2.0 * _contraction(info, viscous)


def test_mixed_degree_count_is_the_uniform_one_for_equal_degrees():
    both = w.flops_per_element(NS3, True, "assemble") + w.flops_per_element(NS3, True, "condense")
    assert w.class_flops_per_element(3, 3, 200) == pytest.approx(both, rel=1e-14)


def test_point_tensor_bytes():
    # 312 and 119 values a volume and face point in 3D with the viscous part, 60 and 36 in 2D without it
    assert w.algorithmic_bytes_per_element(NS3, True, "mixed_assemble") == 8 * (64 * 312 + 64 * 119 + 300 ** 2)
    assert w.algorithmic_bytes_per_element(EU2, False, "mixed_assemble") == 8 * (9 * 60 + 9 * 36 + 60 ** 2)
