"""Standardised face features against NumPy: every face's two one-sided jumps and its last two updates, with a batch that
is no multiple of a block and one that is longer than the grid. FP64 until the last rounding: one FP32 ulp."""
import numpy as np
import pytest

from hdg_cases import Case, GpuCase

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p", [(3, 2), (5, 3), (96, 3)])
def test_features_match_numpy(n, p):
    from oracle.mesh import Mesh
    case = Case("f", 2, n, p, 4.0, 0.5, 0.0, 0.71, "vortex", noise=0.0)
    gc = GpuCase(case)
    torch, hdg, i = gc.torch, gc.hdg, gc.info
    E, F, per, m = i["n_elem"], i["n_faces"], i["Nf"] * i["m"], i["m"]
    rng = np.random.default_rng(n)
    ve = rng.normal(size=(E, m))                                  # constant over an element's nodes
    V = np.repeat(ve[:, None, :], i["Np"], axis=1)
    vh, d1, d2 = (rng.normal(size=(F, i["Nf"], m)) for _ in range(3))
    mean = rng.normal(size=4 * per).astype(np.float32)
    std = (0.5 + rng.random(4 * per)).astype(np.float32)
    mean[per:2 * per], std[per:2 * per] = mean[:per], std[:per]   # both sides alike: their order is the mesh's
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(gc.dev)
    feat = torch.empty((F, 4 * per), dtype=torch.float32, device=gc.dev)
    hdg.hdg_mlp_features(gc.ctx.handle, dev(V), dev(vh), dev(d1), dev(d2), dev(mean), dev(std), feat)
    out = feat.cpu().numpy().astype(np.float64)
    sides = [[] for _ in range(F)]
    for e, faces in enumerate(Mesh(2, n, 0.0, 4.0, p).face_of):
        for f in faces:
            sides[f].append(ve[e])
    jump = np.array(sides)[:, :, None, :] - vh[:, None]           # [F][2][Nf][m]
    ref = (jump.reshape(F, 2, per) - mean[:per].astype(np.float64)) / std[:per]
    scale = (np.abs(jump).reshape(F, 2, per) + np.abs(mean[:per])) / std[:per]
    order = np.argsort(ref, axis=1)                               # each value with its own scale
    ref, scale = np.take_along_axis(ref, order, 1), np.take_along_axis(scale, order, 1)
    assert (np.abs(np.sort(out[:, :2 * per].reshape(F, 2, per), axis=1) - ref) <= 2.0 ** -23 * scale).all()
    for k, d in ((2, d1), (3, d2)):
        mu, s = mean[k * per:(k + 1) * per].astype(np.float64), std[k * per:(k + 1) * per]
        x = d.reshape(F, per)
        assert (np.abs(out[:, k * per:(k + 1) * per] - (x - mu) / s) <= 2.0 ** -23 * (np.abs(x) + np.abs(mu)) / s).all()
