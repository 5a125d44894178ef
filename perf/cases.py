"""The work that users of the library have it do, as measurable cases.

A case is one call (or one short sequence of calls) of the C-ABI binding on a synthetic flow of
the kind the library's own workloads use: periodic boxes of triangles or tetrahedra with edge
length as in those workloads, isentropic vortices in 2D and the Taylor-Green vortex in 3D, the
BDF2 time term with dt = 0.01. Kinds:

  assemble   hdg_assemble_condense, the hot path: every Newton iteration calls it once
  step       hdg_newton_step, a whole implicit time step
  trace      hdg_trace_solve of the condensed system (restarted GMRES)
  matvec     hdg_trace_matvec, the condensed operator on a trace vector (a caller's own solver)
  recover    hdg_recover_interior after a trace solve
  train      hdg_mlp_train_step of the warm-start network on the faces of one time level
  predict    hdg_mlp_features, hdg_mlp_forward and hdg_mlp_apply_trace: the learned trace guess

exact() evaluates the same discrete equations in plain torch FP64: basis, rules and fluxes are
written out here from their definitions, Jacobians come from forward-mode differentiation.
"""
from __future__ import annotations

import itertools
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1808_05066_gb300 import hdg

DEV = torch.device("cuda", 0)
GAMMA = 1.4
DT = 0.01
FP64, MIXED = "fp64", "mixed"


# ------------------------------------------------------------------------------- the cases
def _flow(kind, dim, n, p, **more):
    c = {"kind": kind, "dim": dim, "n": n, "p": p, "viscous": True, "precision": FP64, "scheme": "hdg"}
    if dim == 2:
        c.update(mach=0.5, reynolds=5000.0)
    else:
        c.update(mach=0.1, reynolds=1600.0)
    c.update(more)
    return c


def listed():
    return [
        # the smallest whole call: one implicit step of the 2D Euler vortex on 128 triangles, the
        # size one develops and debugs with; the trace system is small enough for the dense solver
        dict(_flow("step", 2, 8, 2, viscous=False, reynolds=0.0), name="step_euler2d_p2_n8"),
        # a production 2D time step: 32,768 triangles, mixed precision, GMRES trace solves
        dict(_flow("step", 2, 128, 3, precision=MIXED), name="step_ns2d_p3_n128_mixed"),
        # 2D high-order linearisation in plain FP64 on 8,192 triangles
        dict(_flow("assemble", 2, 64, 4, mach=0.3, reynolds=1000.0), name="assemble_ns2d_p4_n64_fp64"),
        # the headline: 82,944 tetrahedra at p = 3, mixed precision; the largest call
        dict(_flow("assemble", 3, 24, 3, precision=MIXED), name="assemble_ns3d_p3_n24_mixed"),
        # the same call on an odd, small mesh (750 elements): a coarse run or one of many subdomains
        dict(_flow("assemble", 3, 5, 3, precision=MIXED), name="assemble_ns3d_p3_n5_mixed"),
        # the plain FP64 form in 3D, the accuracy reference that users compare with
        dict(_flow("assemble", 3, 8, 3), name="assemble_ns3d_p3_n8_fp64"),
        # p-adaptive meshes: degrees 1..4 per element in one persistent launch
        dict(_flow("assemble", 3, 8, 4, degrees="mixed"), name="assemble_ns3d_degrees_n8_fp64"),
        # the linear solve between two linearisations
        dict(_flow("trace", 3, 8, 3), name="trace_solve_ns3d_p3_n8"),
        # the condensed operator and the interior recovery: one pass over S, one over X
        dict(_flow("matvec", 3, 12, 3), name="trace_matvec_ns3d_p3_n12"),
        dict(_flow("recover", 3, 12, 3), name="recover_ns3d_p3_n12"),
        # training and using the warm-start network on the 49,152 faces of the 128 x 128 workload
        {"name": "train_mlp_64_49152", "kind": "train", "net": 64, "batch": 49152},
        dict(_flow("predict", 2, 128, 3), name="predict_ns2d_p3_n128"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# assemble: (dim, p, viscous, precision) with the range of cells per axis
_ASSEMBLE = [
    (2, 1, False, FP64, 8, 160), (2, 2, False, FP64, 8, 128), (2, 2, False, MIXED, 8, 160), (2, 3, False, FP64, 8, 96),
    (2, 2, True, FP64, 8, 128), (2, 3, True, FP64, 8, 96), (2, 3, True, MIXED, 8, 160), (2, 4, True, FP64, 8, 80),
    (2, 4, True, MIXED, 8, 96), (3, 1, True, FP64, 3, 20), (3, 1, True, MIXED, 3, 24), (3, 2, True, FP64, 3, 12),
    (3, 2, True, MIXED, 3, 20), (3, 3, True, FP64, 2, 9), (3, 3, True, MIXED, 2, 18),
]


def draw(rng):
    """A case of the same ranges that is none of the listed ones."""
    have = [{k: v for k, v in c.items() if k != "name"} for c in listed()]
    while (c := _drawn(rng)) in have:
        pass
    return c


def _drawn(rng):
    kind = rng.choice(["assemble"] * 5 + ["degrees", "step", "step", "trace", "matvec", "recover", "train", "predict"])
    if kind == "assemble":
        dim, p, visc, prec, lo, hi = rng.choice(_ASSEMBLE)
        more = {} if visc else {"viscous": False, "reynolds": 0.0}
        return _flow("assemble", dim, _log_int(rng, lo, hi), p, precision=prec, **more)
    if kind == "degrees":
        return _flow("assemble", 3, _log_int(rng, 2, 9), 4, degrees="mixed")
    if kind == "step":
        which = rng.randrange(4)
        if which == 0:  # dense trace solves, each trace space
            return _flow("step", 2, rng.randrange(4, 10), 2, viscous=False, reynolds=0.0,
                         scheme=rng.choice(["hdg", "edg"]))
        if which == 1:
            return _flow("step", 2, _log_int(rng, 18, 96), rng.choice([2, 3]), scheme=rng.choice(["hdg", "edg"]))
        if which == 2:
            return _flow("step", 2, _log_int(rng, 16, 128), 3, precision=MIXED)
        return _flow("step", 3, _log_int(rng, 3, 8), rng.choice([1, 2, 3]), precision=MIXED)
    if kind == "trace":
        return _flow("trace", 3, _log_int(rng, 4, 10), rng.choice([1, 2, 3]))
    if kind in ("matvec", "recover"):
        dim = rng.choice([2, 3])
        n = _log_int(rng, 16, 160) if dim == 2 else _log_int(rng, 4, 15)
        return _flow(kind, dim, n, rng.choice([2, 3]))
    if kind == "train":
        return {"kind": "train", "net": rng.choice([48, 64]), "batch": _log_int(rng, 700, 200000)}
    return _flow("predict", 2, _log_int(rng, 16, 160), rng.choice([2, 3]))


# ------------------------------------------------------------------------------- the inputs
def _box(case):
    return 1.25 * case["n"] if case["dim"] == 2 else 2.0 * math.pi


def _rng(seed, salt):
    return np.random.Generator(np.random.PCG64([seed, salt]))


def _primitives(case, seed, x):
    """(rho, velocity, p) at the points x [..., dim]: seeded vortices or a shifted Taylor-Green state."""
    rng, L, mach = _rng(seed, 1), _box(case), case["mach"]
    x = torch.as_tensor(x, dtype=torch.float64, device=DEV)
    if case["dim"] == 3:
        X, Y, Z = (x + torch.as_tensor(rng.uniform(0, L, 3), device=DEV)).unbind(-1)
        vel = torch.stack([X.sin() * Y.cos() * Z.cos(), -X.cos() * Y.sin() * Z.cos(), torch.zeros_like(X)], -1)
        p = 1.0 / (GAMMA * mach ** 2) + ((2 * X).cos() + (2 * Y).cos()) * ((2 * Z).cos() + 2.0) / 16.0
        rho = torch.ones_like(X)
    else:  # one isentropic vortex per 5 lengths of box (16 on 80 x 80), strengths U[1, 5]
        count = max(1, round(L / 5.0)) if L > 20.0 else 1
        h = torch.ones_like(x[..., 0])
        vel = torch.zeros_like(x)
        phase = 2 * math.pi * (x / L + torch.as_tensor(rng.uniform(0, 1, 2), device=DEV))
        vel[..., 0] = 1.0 + 0.02 * phase[..., 1].sin()  # a weak shear between the vortices
        vel[..., 1] = 0.02 * phase[..., 0].sin()
        side = math.ceil(math.sqrt(count))  # centres in separate cells of a coarse grid, clear of each other
        cells = rng.permutation(side * side)[:count]
        at = (np.stack([cells % side, cells // side], -1) + 0.5 + rng.uniform(-0.2, 0.2, (count, 2))) * (L / side)
        for (cx, cy), psi in zip(at, rng.uniform(1, 5, count)):
            d = x - torch.tensor([cx, cy], dtype=torch.float64, device=DEV)
            d = d - L * torch.round(d / L)
            e1 = (1.0 - d.square().sum(-1)).exp()
            vel[..., 0] -= psi / (2 * math.pi) * e1 * d[..., 1]
            vel[..., 1] += psi / (2 * math.pi) * e1 * d[..., 0]
            h -= (GAMMA - 1.0) * mach ** 2 * psi ** 2 * e1 * e1 / (16.0 * math.pi ** 2)
        rho = h ** (1.0 / (GAMMA - 1.0))
        p = rho ** GAMMA / (GAMMA * mach ** 2)
    return rho, vel, p


def _entropy(case, seed, x):
    """Entropy variables of the flow at the points x."""
    rho, vel, p = _primitives(case, seed, x)
    g1 = GAMMA - 1.0
    s = p.log() - GAMMA * rho.log()
    rho_e = p / g1 + 0.5 * rho * vel.square().sum(-1)
    v1 = -s + GAMMA + 1.0 - g1 * rho_e / p
    return torch.cat([v1[..., None], (g1 * rho / p)[..., None] * vel, (-g1 * rho / p)[..., None]], -1).contiguous()


def _noise(v, eps, gen):
    """Additive noise scaled per component, so that no face point sits on the kink of |V . n|."""
    s = v.reshape(-1, v.shape[-1]).abs().amax(0)
    s[1:-1] = s[1:-1].max()
    return v + eps * s * (2.0 * torch.rand(v.shape, generator=gen, dtype=torch.float64, device=DEV) - 1.0)


def _elements(case):
    return (2 if case["dim"] == 2 else 6) * case["n"] ** case["dim"]


def _flow_state(case, seed):
    """Mesh, context and level-n state, as a program holds them between time steps."""
    dim, scheme = case["dim"], {"hdg": hdg.HDG_SCHEME_HDG, "edg": hdg.HDG_SCHEME_EDG}[case["scheme"]]
    degrees = None
    if case.get("degrees"):
        degrees = _rng(4, 2).choice([1, 2, 3, 4], size=_elements(case), p=[0.1, 0.3, 0.4, 0.2]).astype(np.int8)
    s = SimpleNamespace(case=case)
    s.mesh = hdg.Mesh(dim, case["n"], 0.0, _box(case), case["p"], p_per_elem=degrees, scheme=scheme)
    s.ctx = hdg.Context(s.mesh, GAMMA, case["mach"], case["reynolds"], 0.71)
    s.info = s.mesh.info
    xnode, xtrace, _ = s.mesh.coords()
    gen = torch.Generator(device=DEV).manual_seed(seed)
    s.V = _entropy(case, seed, xnode)
    s.Vhat = _entropy(case, seed, xtrace)
    if case["kind"] != "step" or dim == 3:  # a time step starts from the state itself; V_z vanishes in 3D
        s.Vhat = _noise(s.Vhat, 1e-3, gen)
    return s, gen


def _linearisation(s, precision):
    """BDF2 history with u^{n-1} = u^n and the output buffers of an assembly."""
    i, f64 = s.info, dict(dtype=torch.float64, device=DEV)
    s.hist = torch.empty_like(s.V)
    hdg.hdg_history(s.ctx.handle, s.V, s.V, 2.0 / DT, -0.5 / DT, s.hist)
    s.mass_coef, s.precision = 1.5 / DT, hdg.HDG_PREC_MIXED if precision == MIXED else hdg.HDG_PREC_FP64
    s.S, s.g = torch.empty(i["len_S"], **f64), torch.empty(i["len_g"], **f64)
    s.recov, s.R = torch.empty(i["len_recov"], **f64), torch.empty(i["len_R"], **f64)
    s.status = torch.zeros(i["n_elem"], dtype=torch.int32, device=DEV)


def _assemble(s):
    hdg.hdg_assemble_condense(s.ctx.handle, s.V, s.Vhat, s.hist, s.mass_coef, s.precision, s.S, s.g, s.recov, s.R,
                              s.status)


def _network(nin, seed, gen):
    """A network in mid-training: initial weights, Adam moments of the size they have then."""
    nh, nout = (64, 16) if nin == 64 else (32, 12)
    P = hdg.hdg_mlp_param_count(nin, nh, nout)
    params = torch.empty((14 * P + 3) // 4, dtype=torch.float32, device=DEV)
    hdg.hdg_mlp_init(params, nin, nh, nout, seed)
    params[P:2 * P] = 1e-3 * torch.randn(P, generator=gen, device=DEV)
    params[2 * P:3 * P] = 1e-6 * (0.5 + torch.rand(P, generator=gen, device=DEV))
    return SimpleNamespace(nin=nin, nh=nh, nout=nout, P=P, params=params)


def prepare(case, seed):
    if case["kind"] == "train":
        gen = torch.Generator(device=DEV).manual_seed(seed)
        s = SimpleNamespace(case=case, net=_network(case["net"], seed, gen))
        s.x = torch.randn((case["batch"], s.net.nin), generator=gen, device=DEV)
        s.target = torch.randn((case["batch"], s.net.nout), generator=gen, device=DEV)
        s.grad = torch.empty(s.net.P, dtype=torch.float32, device=DEV)
        s.loss = torch.empty(1, dtype=torch.float32, device=DEV)
        return s
    s, gen = _flow_state(case, seed)
    i, f64 = s.info, dict(dtype=torch.float64, device=DEV)
    if case["kind"] == "assemble":
        _linearisation(s, case["precision"])
    elif case["kind"] == "step":
        s.precision = hdg.HDG_PREC_MIXED if case["precision"] == MIXED else hdg.HDG_PREC_FP64
    elif case["kind"] == "trace":
        _linearisation(s, FP64)
        _assemble(s)
        s.dVhat = torch.empty(i["n_trace"], **f64)
    elif case["kind"] == "matvec":
        s.S = torch.randn(i["len_S"], generator=gen, **f64)
        s.x = torch.randn(i["n_trace"], generator=gen, **f64)
        s.y = torch.empty(i["n_trace"], **f64)
    elif case["kind"] == "recover":
        s.recov = torch.randn(i["len_recov"], generator=gen, **f64)
        s.dVhat = torch.randn(i["n_trace"], generator=gen, **f64)
        s.dV = torch.empty(i["len_V"], **f64)
    else:  # predict: the last two trace updates, the statistics of the training set
        nt = s.Vhat.shape
        s.net = _network(4 * i["Nf"] * i["m"], seed, gen)
        s.dv1 = 1e-3 * torch.randn(nt, generator=gen, **f64)
        s.dv2 = 1e-3 * torch.randn(nt, generator=gen, **f64)
        s.mean = 1e-4 * torch.randn(s.net.nin, generator=gen, device=DEV)
        s.std = 1e-2 * (0.5 + torch.rand(s.net.nin, generator=gen, device=DEV))
        s.tmean = 1e-5 * torch.randn(s.net.nout, generator=gen, device=DEV)
        s.tstd = 1e-4 * (0.5 + torch.rand(s.net.nout, generator=gen, device=DEV))
        s.feat = torch.empty((i["n_faces"], s.net.nin), dtype=torch.float32, device=DEV)
        s.pred = torch.empty((i["n_faces"], s.net.nout), dtype=torch.float32, device=DEV)
        s.guess = torch.empty_like(s.Vhat)
    return s


# ------------------------------------------------------------------------------- one pass
def run(s):
    kind = s.case["kind"]
    if kind == "assemble":
        _assemble(s)
        return {"S": s.S, "g": s.g, "recov": s.recov, "R": s.R, "status": s.status}
    if kind == "step":  # the first step of a run is BDF1 from the level-n state
        V, Vhat = s.V.clone(), s.Vhat.clone()
        updates, _ = hdg.hdg_newton_step(s.ctx.handle, V, Vhat, s.V, None, DT, 1, s.precision, 1e-10, 10)
        return {"V": V, "Vhat": Vhat, "updates": updates}
    if kind == "trace":
        hdg.hdg_trace_solve(s.ctx.handle, s.S, s.g, s.dVhat, hdg.HDG_SOLVER_GMRES, 1e-12, 600)
        return {"dVhat": s.dVhat}
    if kind == "matvec":
        hdg.hdg_trace_matvec(s.ctx.handle, s.S, s.x, s.y)
        return {"y": s.y}
    if kind == "recover":
        hdg.hdg_recover_interior(s.ctx.handle, s.recov, s.dVhat, s.dV)
        return {"dV": s.dV}
    net = s.net
    if kind == "train":
        hdg.hdg_mlp_train_step(net.params, s.grad, net.nin, net.nh, net.nout, s.x, s.target, s.case["batch"], 1e-3,
                               100, s.loss)
        P = net.P
        return {"grad": s.grad, "loss": s.loss, "params": net.params[:P], "m": net.params[P:2 * P],
                "v": net.params[2 * P:3 * P], "bf16": net.params[3 * P:].view(torch.bfloat16)[:P]}
    hdg.hdg_mlp_features(s.ctx.handle, s.V, s.Vhat, s.dv1, s.dv2, s.mean, s.std, s.feat)
    hdg.hdg_mlp_forward(net.params, net.nin, net.nh, net.nout, s.feat, s.info["n_faces"], s.pred)
    hdg.hdg_mlp_apply_trace(s.ctx.handle, s.Vhat, s.dv1, s.pred, s.tmean, s.tstd, s.guess)
    return {"feat": s.feat, "pred": s.pred, "guess": s.guess}


# ------------------------------------------------------------------------------- its work
def _sizes(dim, pk, pt):
    m, c = dim + 2, math.comb
    NP, NF = c(pk + dim, dim), dim + 1
    return SimpleNamespace(m=m, NP=NP, NF=NF, Nf=c(pt + dim - 1, dim - 1), NV=NP * m,
                           NT=NF * c(pt + dim - 1, dim - 1) * m, NG=(pk + 1) ** dim, NGF=(pt + 1) ** (dim - 1))


def _element_work(dim, pk, pt):
    """(values in, values out, flops) of one element's linearisation and condensation: one product
    per quadrature point, test function and trial function of each pair of components, the
    factorisation, the solves and the Schur product."""
    z = _sizes(dim, pk, pt)
    nz = z.NP + z.NF * z.Nf
    flops = 2.0 * z.m ** 2 * (z.NP * nz * z.NG + z.NF * z.Nf * nz * z.NGF)
    flops += 2.0 * (z.NV ** 3 / 3.0 + (z.NT + 1) * z.NV ** 2 + (z.NT + 1) * z.NT * z.NV)
    return 2 * z.NV + z.NT / 2, z.NT ** 2 + z.NT + z.NV * z.NT + z.NV + z.NV + z.NT, flops


def work(case):
    kind = case["kind"]
    if kind == "train":
        P = {64: 9360, 48: 3020}[case["net"]]
        nout = {64: 16, 48: 12}[case["net"]]
        return {"bytes": 4.0 * case["batch"] * (case["net"] + nout) + 2 * 14.0 * P, "flops": 6.0 * case["batch"] * P}
    dim, p, E = case["dim"], case["p"], _elements(case)
    z = _sizes(dim, p, p)
    faces = E * z.NF / 2
    if kind in ("assemble", "step", "trace") and case.get("degrees"):
        parts = [(w, _element_work(dim, q, q)) for q, w in zip((1, 2, 3, 4), (0.1, 0.3, 0.4, 0.2))]
        vin, vout, flops = (E * sum(w * e[k] for w, e in parts) for k in range(3))
    else:
        vin, vout, flops = (E * v for v in _element_work(dim, p, p))
    if kind == "assemble":
        return {"bytes": 8.0 * (vin + vout), "flops": flops}
    if kind == "step":  # at least one linearisation
        return {"bytes": 8.0 * (2 * vin + 2 * E * z.NV), "flops": flops}
    if kind == "trace":  # at least one product with every S
        return {"bytes": 8.0 * (E * z.NT * (z.NT + 1) + faces * z.Nf * z.m), "flops": 2.0 * E * z.NT ** 2}
    if kind == "matvec":
        return {"bytes": 8.0 * (E * z.NT ** 2 + 2 * faces * z.Nf * z.m), "flops": 2.0 * E * z.NT ** 2}
    if kind == "recover":
        return {"bytes": 8.0 * (E * (z.NV * z.NT + 2 * z.NV) + faces * z.Nf * z.m), "flops": 2.0 * E * z.NV * z.NT}
    P, nin = (9360, 64) if p == 3 else (3020, 48)
    return {"bytes": 8.0 * (E * z.NV + 4 * faces * nin / 4) + 4.0 * faces * nin * 1.25, "flops": 2.0 * faces * P}


# ------------------------------------------------------------------------------- 64-bit values
def _jacobi_rule(n, a):
    """Gauss-Jacobi points and weights on [0, 1] for the weight (1 - x)^a, from the recurrence's matrix."""
    k = np.arange(n)
    diag = np.where(2 * k + a == 0, 0.0, -a * a / np.maximum((2 * k + a) * (2 * k + a + 2), 1))
    diag[0] = -a / (a + 2)
    k = np.arange(1, n)
    off = np.sqrt(4.0 * k * (k + a) * k * (k + a) / ((2 * k + a) ** 2 * (2 * k + a + 1) * (2 * k + a - 1)))
    x, q = np.linalg.eigh(np.diag(diag) + np.diag(off, 1) + np.diag(off, -1))
    return (1 + x) / 2, q[0] ** 2 / (a + 1)


def _simplex_rule(dim, n):
    """Collapsed rule on the unit simplex, points with the first coordinate fastest."""
    rules = [_jacobi_rule(n, a) for a in range(dim)]
    pts, wts = [], []
    for ix in itertools.product(range(n), repeat=dim):  # last coordinate slowest
        left, x, w = 1.0, [0.0] * dim, 1.0
        for r in reversed(range(dim)):
            t, wt = rules[r][0][ix[dim - 1 - r]], rules[r][1][ix[dim - 1 - r]]
            x[r], left, w = t * left, (1 - t) * left, w * wt
        pts.append(x)
        wts.append(w)
    return np.array(pts), np.array(wts)


class _Basis:
    """Nodal P_p basis on the equispaced lattice, through the inverse of a monomial Vandermonde matrix."""

    def __init__(self, dim, p):
        self.ix = np.array([ix[::-1] for ix in itertools.product(range(p + 1), repeat=dim) if sum(ix) <= p])
        self.faces = [np.flatnonzero(self.ix.sum(1) == p)] + [np.flatnonzero(self.ix[:, r] == 0) for r in range(dim)]
        self.nodes = self.ix / p
        self.inv = np.linalg.inv(self._mono(self.nodes, self.ix))

    @staticmethod
    def _mono(x, ex):
        return np.prod(x[:, None, :] ** ex[None], -1)

    def values(self, x):
        return self._mono(x, self.ix) @ self.inv

    def gradients(self, x):
        out = []
        for r in range(x.shape[1]):
            ex = self.ix.copy()
            ex[:, r] = np.maximum(ex[:, r] - 1, 0)
            out.append((self._mono(x, ex) * self.ix[:, r]) @ self.inv)
        return np.stack(out, -1)


def _t(x):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64, device=DEV)


class _Element:
    """The local residuals of elements of degree pk whose trace is given in degree pt on every face."""

    def __init__(self, case, pk, pt):
        dim = self.dim = case["dim"]
        self.mach, self.reynolds = case["mach"], case["reynolds"] if case["viscous"] else 0.0
        b, bt = _Basis(dim, pk), _Basis(dim, pt)
        x, w = _simplex_rule(dim, pk + 1)
        xf, wf = _simplex_rule(dim - 1, pt + 1)
        verts = np.vstack([np.zeros(dim), np.eye(dim)])
        self.w, self.phi, self.dphi = _t(w), _t(b.values(x)), _t(b.gradients(x))
        mass_inv = np.linalg.inv(b.values(x).T @ (w[:, None] * b.values(x)))
        phif, dphif, psi, lift = [], [], [], []
        for f in range(dim + 1):
            y = np.delete(verts, f, 0)
            pts = y[0] + xf @ (y[1:] - y[0])
            phif.append(b.values(pts))
            dphif.append(b.gradients(pts))
            psi.append(bt.values(pts)[:, bt.faces[f]])
            lift.append(mass_inv @ (phif[-1].T * wf))      # face-point values -> nodal lift coefficients
        self.wf, self.phif, self.dphif = _t(wf), _t(np.stack(phif)), _t(np.stack(dphif))
        self.psi, self.lift = _t(np.stack(psi)), _t(np.stack(lift))

    def _prim(self, v):
        vm = v[..., -1]
        s = GAMMA - v[..., 0] + v[..., 1:-1].square().sum(-1) / (2.0 * vm)
        rho = ((math.log(GAMMA - 1.0) - (-vm).log() - s) / (GAMMA - 1.0)).exp()
        return rho, -v[..., 1:-1] / vm[..., None], -rho * (GAMMA - 1.0) / vm

    def _u(self, v):
        rho, vel, p = self._prim(v)
        e = p / (GAMMA - 1.0) + 0.5 * rho * vel.square().sum(-1)
        return torch.cat([rho[..., None], rho[..., None] * vel, e[..., None]], -1)

    def _flux(self, v):
        rho, vel, p = self._prim(v)
        H = p / (GAMMA - 1.0) + 0.5 * rho * vel.square().sum(-1) + p
        mom = rho[..., None, None] * vel[..., :, None] * vel[..., None, :]
        mom = mom + p[..., None, None] * torch.eye(self.dim, dtype=v.dtype, device=v.device)
        return torch.cat([(rho[..., None] * vel)[..., None, :], mom, (H[..., None] * vel)[..., None, :]], -2)

    def _viscous(self, v, q):
        vm = v[..., -1]
        cv, mu = 1.0 / (GAMMA * (GAMMA - 1.0) * self.mach ** 2), 1.0 / self.reynolds
        kappa = GAMMA * cv * mu / 0.71
        vel = -v[..., 1:-1] / vm[..., None]
        gv = v[..., 1:-1, None] * q[..., -1:, :] / (vm * vm)[..., None, None] - q[..., 1:-1, :] / vm[..., None, None]
        div = torch.diagonal(gv, dim1=-2, dim2=-1).sum(-1)
        eye = torch.eye(self.dim, dtype=v.dtype, device=v.device)
        tau = mu * (gv + gv.transpose(-1, -2) - (2.0 / 3.0) * div[..., None, None] * eye)
        e = (vel[..., :, None] * tau).sum(-2) + kappa * q[..., -1, :] / (cv * vm * vm)[..., None]
        return -torch.cat([torch.zeros_like(e)[..., None, :], tau, e[..., None, :]], -2)

    def _face_flux(self, vh, v, n):
        rho, vel, p = self._prim(vh)
        lam = (vel * n).sum(-1).abs() + (GAMMA * p / rho).sqrt()
        du = torch.func.jvp(self._u, (vh,), (v - vh,))[1]        # A0(vhat) (v - vhat)
        f = ((self._flux(vh) + self._flux(v)) * n[..., None, :]).sum(-1)
        return 0.5 * (f + lam[..., None] * du)

    def residuals(self, v, vhq, jinv, det, pro, mass_coef, hist):
        """R_v [NP, m] and R_t (in the faces' own spaces) of one element."""
        vh = torch.einsum("fcq,fqi->fci", pro, vhq)
        # q = grad v + lift of the face jumps; n |F| / |K| per face in terms of the rows of jinv
        ns = -torch.cat([-jinv.sum(0, keepdim=True), jinv], 0)   # outward n s_F / |det J|
        jump = torch.einsum("fgc,fci->fgi", self.psi, vh) - torch.einsum("fgb,bi->fgi", self.phif, v)
        lifted = torch.einsum("fbg,fgi->fbi", self.lift, jump)   # nodal values, per face
        qn = torch.einsum("fbi,fk->bik", lifted, ns)

        def q_at(phi, dphi):
            return torch.einsum("gbr,rk,bi->gik", dphi, jinv, v) + torch.einsum("gb,bik->gik", phi, qn)

        vg = self.phi @ v
        F = self._flux(vg)
        if self.reynolds:
            F = F + self._viscous(vg, q_at(self.phi, self.dphi))
        W = self.w * det
        Rv = mass_coef * torch.einsum("g,ga,gi->ai", W, self.phi, self._u(vg)) - hist
        Rv = Rv - torch.einsum("g,gar,rk,gik->ai", W, self.dphi, jinv, F)
        Rt = []
        for f in range(self.dim + 1):
            size = ns[f].norm()
            n, Wf = ns[f] / size, self.wf * det * size
            vf, vhf = self.phif[f] @ v, self.psi[f] @ vh[f]
            h = self._face_flux(vhf, vf, n.expand(vf.shape[0], self.dim))
            if self.reynolds:
                h = h + (self._viscous(vhf, q_at(self.phif[f], self.dphif[f])) * n).sum(-1)
            Rv = Rv + torch.einsum("g,gb,gi->bi", Wf, self.phif[f], h)
            Rt.append(pro[f].T @ torch.einsum("g,gc,gi->ci", Wf, self.psi[f], h))
        return Rv, torch.stack(Rt)

    def blocks(self, v, vh, jinv, det, pro, mass_coef, hist):
        """(R_v, R_t, A, B, C, D) of a batch of elements."""
        NV, NT = v[0].numel(), vh[0].numel()

        def flat(z, *geo):
            Rv, Rt = self.residuals(z[:NV].view(v.shape[1:]), z[NV:].view(vh.shape[1:]), *geo[:3], mass_coef, geo[3])
            r = torch.cat([Rv.reshape(-1), Rt.reshape(-1)])
            return r, r

        z = torch.cat([v.flatten(1), vh.flatten(1)], 1)
        J, R = torch.func.vmap(torch.func.jacfwd(flat, has_aux=True))(z, jinv, det, pro, hist)
        return R[:, :NV], R[:, NV:], J[:, :NV, :NV], J[:, :NV, NV:], J[:, NV:, :NV], J[:, NV:, NV:]


def _condensed(s, V, Vhat, hist, mass_coef):
    """The outputs of the linearisation, element groups of one class at a time: a list of
    (elements, own trace unknowns, S, g, X, y, R_v, R_t)."""
    case, i = s.case, s.info
    dim, m, nF, Nfm = case["dim"], i["m"], i["nF"], i["Nf"]
    E = i["n_elem"]
    lay = s.mesh.layout()
    face_of = s.mesh.topology()[0]
    fdeg = lay["face_deg"][face_of].astype(int)
    tn = torch.as_tensor(s.mesh.trace_map().astype(np.int64), device=DEV)
    pk, pt = lay["elem_p"].astype(int), fdeg.max(1)
    Vf, Hf, Vh = V.reshape(-1), hist.reshape(-1), Vhat.reshape(-1, m)
    xn = s.mesh.coords()[0].reshape(-1, dim)
    out = []
    for k, t in sorted(set(zip(pk.tolist(), pt.tolist()))):
        el = _Element(case, k, t)
        b = _Basis(dim, k)
        ids = np.flatnonzero((pk == k) & (pt == t))
        corner = [int(np.flatnonzero((b.nodes == c).all(1))[0]) for c in np.vstack([np.zeros(dim), np.eye(dim)])]
        pros = {}                                              # degree q -> degree t, padded to the widest face
        for q in range(1, t + 1):
            bq, bt = _Basis(dim, q), _Basis(dim, t)
            P = np.zeros((nF, len(bt.faces[0]), Nfm))
            for f in range(nF):
                P[f, :, :len(bq.faces[f])] = bq.values(bt.nodes[bt.faces[f]])[:, bq.faces[f]]
            pros[q] = _t(P)
        step = max(1, int(4e8 / (8.0 * (len(b.ix) + nF * Nfm) * m * (len(el.w) + nF * len(el.wf)) * m * dim)))
        for c0 in range(0, len(ids), step):
            e = ids[c0:c0 + step]
            nodes = (lay["voff"][e] // m)[:, None] + np.arange(len(b.ix))
            X = xn[nodes[:, corner]]                           # vertices
            jac = np.swapaxes(X[:, 1:] - X[:, :1], 1, 2)       # dx / dr
            jinv, det = _t(np.linalg.inv(jac)), _t(np.abs(np.linalg.det(jac)))
            idx = torch.as_tensor(nodes, device=DEV)
            v, h = Vf.view(-1, m)[idx], Hf.view(-1, m)[idx]
            own = tn[e]
            vh = torch.where((own >= 0)[..., None], Vh[own.clamp(min=0)], 0.0)
            pro = torch.stack([torch.stack([pros[q][f] for f, q in enumerate(r)]) for r in fdeg[e].tolist()])
            Rv, Rt, A, B, C, D = el.blocks(v, vh, jinv, det, pro, mass_coef, h)
            XY = torch.linalg.solve(A, torch.cat([B, Rv[..., None]], -1))
            Xe, y = XY[..., :-1], XY[..., -1]
            out.append((e, (own >= 0).repeat_interleave(m, -1).flatten(1), D - C @ Xe, Rt - (C @ y[..., None])[..., 0],
                        Xe, y, Rv, Rt))
    return out, lay


def _exact_assemble(s):
    groups, lay = _condensed(s, s.V, s.Vhat, s.hist, s.mass_coef)
    out = {k: torch.empty(s.info["len_" + k], dtype=torch.float64, device=DEV) for k in ("S", "g", "recov", "R")}
    for e, own, S, g, X, y, Rv, Rt in groups:
        for j, ee in enumerate(e.tolist()):
            o = own[j]
            for name, off, val in (("S", "soff", S[j][o][:, o]), ("g", "toff", g[j][o]),
                                   ("recov", "roff", torch.cat([X[j][:, o].reshape(-1), y[j]])),
                                   ("R", "Roff", torch.cat([Rv[j], Rt[j][o]]))):
                out[name][lay[off][ee]:lay[off][ee + 1]] = val.reshape(-1)
    return out | {"status": None}


def _gather_index(s):
    """[E, NT] global trace unknown of each local one."""
    m = s.info["m"]
    tn = torch.as_tensor(s.mesh.trace_map().astype(np.int64), device=DEV)
    return (tn[..., None] * m + torch.arange(m, device=DEV)).flatten(1)


def _exact_step(s):
    """Newton's method with dense trace solves, past the tolerance of the measured call."""
    idx, n = _gather_index(s), s.info["n_trace"]
    el = _Element(s.case, s.case["p"], s.case["p"])
    det = _t(s.mesh.coords()[2][:, s.case["dim"] ** 2])
    mass = 1.0 / DT
    hist = mass * torch.einsum("e,g,ga,egi->eai", det, el.w, el.phi, el._u(torch.einsum("gb,ebi->egi", el.phi, s.V)))
    V, Vhat = s.V.clone(), s.Vhat.clone()
    for _ in range(7):
        K = torch.zeros(n * n, dtype=torch.float64, device=DEV)
        rhs, dV = torch.zeros(n, dtype=torch.float64, device=DEV), torch.empty_like(V)
        groups = _condensed(s, V, Vhat, hist, mass)[0]
        for e, _, S, g, *_ in groups:
            ix = idx[torch.as_tensor(e, device=DEV)]
            K.index_add_(0, (ix[:, :, None] * n + ix[:, None, :]).flatten(), S.flatten())
            rhs.index_add_(0, ix.flatten(), -g.flatten())
        d = torch.linalg.solve(K.view(n, n), rhs)
        for e, _, _, _, X, y, *_ in groups:
            et = torch.as_tensor(e, device=DEV)
            dV[et] = (-y - (X @ d[idx[et]][..., None])[..., 0]).view(len(e), *V.shape[1:])
        V += dV
        Vhat += d.view(Vhat.shape)
    return {"V": V, "Vhat": Vhat, "updates": None}


def _mlp(net, x):
    """Layer outputs of the network with its bf16 weights, and the weights, in FP64."""
    w = net.params[3 * net.P:].view(torch.bfloat16)[:net.P].double()
    shapes = [(net.nh, net.nin), (net.nh,), (net.nh, net.nh), (net.nh,), (net.nout, net.nh), (net.nout,)]
    W1, b1, W2, b2, W3, b3 = (p.view(sh) for p, sh in zip(w.split([math.prod(sh) for sh in shapes]), shapes))
    h1 = torch.tanh(x.double() @ W1.T + b1)
    h2 = torch.tanh(h1 @ W2.T + b2)
    return h1, h2, h2 @ W3.T + b3, W2, W3


def _exact_train(s):
    net, P = s.net, s.net.P
    x = s.x.double()
    h1, h2, y, W2, W3 = _mlp(net, x)
    d = y - s.target.double()
    dy = 2.0 * d / d.numel()
    d2 = dy @ W3 * (1 - h2 * h2)
    d1 = d2 @ W2 * (1 - h1 * h1)
    grad = torch.cat([t.reshape(-1) for t in (d1.T @ x, d1.sum(0), d2.T @ h1, d2.sum(0), dy.T @ h2, dy.sum(0))])
    m = 0.9 * net.params[P:2 * P].double() + 0.1 * grad
    v = 0.999 * net.params[2 * P:3 * P].double() + 0.001 * grad * grad
    p = net.params[:P].double() - 1e-3 * (m / (1 - 0.9 ** 100)) / ((v / (1 - 0.999 ** 100)).sqrt() + 1e-8)
    return {"grad": grad, "loss": d.square().mean().reshape(1), "params": p, "m": m, "v": v, "bf16": None}


def _exact_predict(s):
    i = s.info
    fnodes = np.stack(_Basis(s.case["dim"], s.case["p"]).faces)
    _, fmap, side = s.mesh.topology()
    feats = []
    for k in range(2):  # each side's node values in the face's canonical node order
        e, f = side[:, k] // i["nF"], side[:, k] % i["nF"]
        node = np.take_along_axis(fnodes[f], np.argsort(fmap[e, f], 1), 1)
        feats.append(s.V[torch.as_tensor(e, device=DEV)[:, None], torch.as_tensor(node, device=DEV)] - s.Vhat)
    raw = torch.cat([t.flatten(1) for t in feats + [s.dv1, s.dv2]], 1)
    feat = (raw - s.mean.double()) / s.std.double()
    pred = _mlp(s.net, feat)[2]
    guess = s.Vhat + s.dv1 + (pred * s.tstd.double() + s.tmean.double()).view(s.Vhat.shape)
    return {"feat": feat, "pred": pred, "guess": guess}


def exact(case, seed):
    kind = case["kind"]
    if kind == "assemble" and work(case)["flops"] > 4e11:      # above 20 s
        return None
    if kind == "step" and (case["scheme"] != "hdg" or _elements(case) > 200):
        return None                                            # a dense solve per update: above 20 s
    s = prepare(case, seed)
    if kind == "assemble":
        return _exact_assemble(s)
    if kind == "step":
        return _exact_step(s)
    if kind == "train":
        return _exact_train(s)
    if kind == "predict":
        return _exact_predict(s)
    idx, E = _gather_index(s), s.info["n_elem"]
    nv, nt, n = s.info["nv"], s.info["nt"], s.info["n_trace"]
    if kind == "matvec":
        y = torch.einsum("ers,es->er", s.S.view(E, nt, nt), s.x[idx])
        return {"y": torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, idx.flatten(), y.flatten())}
    if kind == "recover":
        X, y = s.recov.view(E, -1)[:, :nv * nt].view(E, nv, nt), s.recov.view(E, -1)[:, nv * nt:]
        return {"dV": (-y - torch.einsum("ers,es->er", X, s.dVhat[idx])).flatten()}
    if n > 12000:                                              # trace: a dense solve above 20 s
        return None
    K = torch.zeros(n * n, dtype=torch.float64, device=DEV)
    K.index_add_(0, (idx[:, :, None] * n + idx[:, None, :]).flatten(), s.S)
    rhs = torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, idx.flatten(), -s.g)
    return {"dVhat": torch.linalg.solve(K.view(n, n), rhs)}
