"""CPU pins of the two identities behind the FP64 contraction in reference coordinates: the scaled
face normals are constant combinations of the rows of Jinv, and the viscous flux Jacobian contracted
with a vector on both sides has the closed form the pointwise kernel evaluates."""
import numpy as np
import pytest

from oracle import physics as ph
from paper_1808_05066_gb300 import hdg


@pytest.mark.parametrize("dim", [2, 3])
def test_scaled_normals_are_rows_of_jinv(dim):
    mesh = hdg.Mesh(dim, [2, 3, 1][:dim], [0.0, -1.0, 0.5][:dim], [1.0, 3.0, 2.0][:dim], 2)
    geo = mesh.coords()[2]
    jinv = geo[:, :dim * dim].reshape(-1, dim, dim)
    det = geo[:, dim * dim]
    face = geo[:, dim * dim + 1:].reshape(len(geo), dim + 1, dim + 1)
    ns = face[..., :dim] * (face[..., dim] / det[:, None])[..., None]
    expect = np.concatenate([jinv.sum(1, keepdims=True), -jinv], 1)
    assert np.abs(ns - expect).max() <= 1e-14 * np.abs(expect).max()


@pytest.mark.parametrize("d", [2, 3])
def test_pair_contraction_closed_form(d):
    """sum_jk c_j c2_k dG_ij/dq_lk against the oracle's viscous flux at unit gradients."""
    rng = np.random.default_rng(3 + d)
    phys = ph.Physics(gamma=1.4, mach=0.3, reynolds=400.0, prandtl=0.71)
    m = d + 2
    for _ in range(20):
        v = ph.v_of_u(ph.u_of_primitives(np.array(rng.uniform(0.5, 2.0)), rng.normal(size=d),
                                         np.array(rng.uniform(5.0, 9.0)), phys.gamma), phys.gamma)
        c, c2 = rng.normal(size=d), rng.normal(size=d)
        ref = np.zeros((m, m))
        for l in range(m):
            q = np.zeros((m, d))
            q[l] = c2
            ref[:, l] = ph.viscous_flux(v, q, phys) @ c
        ivm = 1.0 / v[-1]
        vel, A = -v[1:-1] * ivm, v[1:-1] * ivm * ivm
        cc, cA, cV, eA, eV, VA = c @ c2, c @ A, c @ vel, c2 @ A, c2 @ vel, vel @ A
        got = np.zeros((m, m))
        got[1:-1, 1:-1] = phys.mu * ivm * (np.outer(c2, c) - (2.0 / 3.0) * np.outer(c, c2) + cc * np.eye(d))
        got[1:-1, -1] = -phys.mu * (A * cc + c2 * cA - (2.0 / 3.0) * eA * c)
        got[-1, 1:-1] = phys.mu * ivm * (vel * cc + eV * c - (2.0 / 3.0) * c2 * cV)
        got[-1, -1] = -phys.mu * (VA * cc + eV * cA - (2.0 / 3.0) * eA * cV) - phys.kappa / phys.cv * ivm ** 2 * cc
        assert np.abs(got - ref).max() <= 1e-13 * np.abs(ref).max()
