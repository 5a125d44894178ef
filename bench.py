#!/usr/bin/env python3
"""Benchmark of the hot path: assemble + condense throughput (elements/s) for 3D
Navier-Stokes tetrahedra at p = 3 — the 24^3 periodic cube [0, 2pi]^3, 6 tets per cell
(82,944 elements; local interior system 400 x 400, reduced to 100 x 100 by the exact
q-elimination; trace block 200 x 200), Taylor-Green initial state at M0 = 0.1,
Re = 1600, Pr = 0.71, trace perturbed by 1e-3, BDF2 time term with dt = 0.01.

One step = one hdg_assemble_condense over all elements (residuals, pointwise Jacobians,
quadrature contractions, LU, X = A^{-1}B, S = D - C X, g). Inputs are resident in HBM;
each step writes S (26.5 GB) and the recovery data (13.3 GB), far more than L2.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--precision fp64|mixed]
  python bench.py --impl reference     # the FP64 CPU oracle on a bounded sample

Prints one JSON line (rank 0).
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

WORKLOAD = "ns3d_p3_tgv"
METRIC = "elem/s assemble+condense (3D NS tet p=3), mixed vs FP64, rel err ≤1e-10"
UNIT = "elem/s"


# ----------------------------------------------------------------------------- oracle pool
_ORACLE = {}


def _oracle_init(n_override):
    """Worker set-up (untimed): the oracle's own mesh and state of the workload."""
    import numpy as np

    import workloads as wl
    from oracle import physics as ph
    from oracle.hdg import Problem, interpolate_state
    from oracle.mesh import Mesh
    spec = dict(wl.WORKLOADS[WORKLOAD])
    if n_override:
        spec["n"] = n_override
    mesh = Mesh(spec["dim"], spec["n"], spec["lo"], spec["hi"], spec["p"])
    phys = ph.Physics(mach=spec["mach"], reynolds=spec["reynolds"], prandtl=spec["prandtl"])
    prob = Problem(mesh, phys)
    V, Vh = interpolate_state(prob, lambda x: wl.primitive_state(WORKLOAD, x, **spec))
    Vh = wl.perturb(Vh, spec["trace_noise"], spec["seed"])
    _ORACLE.update(prob=prob, V=V, Vh=Vh, dt=spec["dt"])


def _oracle_condense(e):
    """Oracle condensation of element e (BDF2 with u^{n-1} = u^n); returns its S norm."""
    import numpy as np
    prob, V, Vh, dt = _ORACLE["prob"], _ORACLE["V"], _ORACLE["Vh"], _ORACLE["dt"]
    vh = prob.gather_trace(Vh, e)
    Q = prob.consistent_q(e, V[e], vh)
    hist = prob.history_weak(e, [V[e], V[e]], [2.0 / dt, -0.5 / dt])
    L = prob.condense(e, Q, V[e], vh, 1.5 / dt, hist)
    return float(np.linalg.norm(L["S"]))


def oracle_throughput(n_elem_total, per_core, steps=1, warmup=0, n_override=None):
    """Time the oracle on a seeded sample of elements in a spawn pool over all host
    cores. Returns (elem/s per step list, cores, sample description)."""
    import multiprocessing as mp

    import numpy as np
    cores = os.cpu_count() or 1
    env_keep = {k: os.environ.get(k) for k in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS")}
    for k in env_keep:
        os.environ[k] = "1"
    ctx = mp.get_context("spawn")
    rates = []
    rng = np.random.default_rng(3)
    try:
        with ctx.Pool(cores, initializer=_oracle_init, initargs=(n_override,)) as pool:
            pool.map(_oracle_condense, [0] * cores)  # pay the set-up in every worker
            sample = rng.choice(n_elem_total, size=cores * per_core, replace=False).tolist()
            for it in range(warmup + steps):
                t0 = time.perf_counter()
                pool.map(_oracle_condense, sample, chunksize=per_core)
                dt = time.perf_counter() - t0
                if it >= warmup:
                    rates.append(len(sample) / dt)
    finally:
        for k, v in env_keep.items():
            if v is None:
                os.environ.pop(k, None)
            else:
                os.environ[k] = v
    desc = (f"{cores * per_core} seeded random elements (one fixed sample) of the {n_elem_total}-element workload, "
            f"oracle condense (complex-step Jacobian, dense 400x400 LU) in a spawn pool of {cores} processes")
    return rates, cores, desc


# ----------------------------------------------------------------------------- clocks
class ClockSampler:
    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits", "-lms", "200",
                 "-i", str(self.gpu)], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except (OSError, FileNotFoundError):
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *exc):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 8:
                continue
            try:
                sm.append(float(parts[0]))
                mx.append(float(parts[1]))
            except ValueError:
                continue
            for nm, val in zip(names, parts[4:8]):
                if val.lower().startswith("active"):
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"], "samples": 0}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


# ----------------------------------------------------------------------------- main
def measured_peaks() -> dict:
    """HBM copy bandwidth and sustained dense bf16 rate measured on this GPU type
    (MEASURED_PEAKS.json beside this file), else the earlier single measurement."""
    path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "MEASURED_PEAKS.json")
    try:
        with open(path) as fh:
            d = json.load(fh)
        return {"hbm": float(d["hbm_gbs"]), "bf16": float(d["bf16_tflops_sustained"]),
                "hbm_source": "measured: STREAM-style copy (MEASURED_PEAKS.json)",
                "bf16_source": "measured: cuBLAS bf16 GEMM, sustained (MEASURED_PEAKS.json)"}
    except (OSError, KeyError, ValueError):
        return {"hbm": 6800.0, "bf16": 1700.0, "hbm_source": "fallback: earlier GB300 measurement",
                "bf16_source": "fallback: earlier GB300 measurement, sustained"}


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--precision", choices=["fp64", "mixed"], default="mixed")
    ap.add_argument("--fp64-steps", type=int, default=2, help="timed steps of the FP64 comparison form")
    ap.add_argument("--cpu-per-core", type=int, default=8, help="oracle elements per host core and step")
    ap.add_argument("--n", type=int, default=None, help="override the cube resolution (tests only)")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-newton", action="store_true", help="skip the Newton-step wall time")
    ap.add_argument("--no-mixed-degree", action="store_true", help="skip the mixed-degree batch")
    ap.add_argument("--mixed-degree-steps", type=int, default=2)
    ap.add_argument("--mixed-degree-newton", action="store_true",
                    help="also time one BDF2 Newton step of the mixed-degree batch")
    return ap.parse_args()


# DRAM bytes (dram__bytes_read.sum + dram__bytes_write.sum) per element of the mixed tensor-core
# kernels from one ncu capture on 1,296 elements (more than L2 holds several times over); traffic
# grows with the element count and scales to a launch by its elements. Valid only while the kernel
# sources hash to the digest they were captured on.
NCU_TRAFFIC = {
    "source": "profiles/ncu_mixed_kernels_ns3d_p3_n6.md",
    "sources_sha256": "5ab3f99d2cf46a6a3abc049d5255352aa8f21e36f33d58df059bbc6bdbbeb8fc",
    "bytes_per_element": {"mixed_assemble": 3_988_032, "mixed_condense": 1_390_173},
}

# the sources that define the captured kernels and their launch shapes (device code and the
# dispatch of the mixed form); host-side entry points do not change the kernels
KERNEL_SOURCES = ("asm_t5.cuh", "condense_tc.cuh", "condense_t5.cuh", "ozaki.cuh", "dfloat.cuh",
                  "element_fp64.cuh", "assemble_fp64.cuh", "hdg_device.cuh", "assemble_mixed.cu")


def kernel_sources_digest() -> str:
    import hashlib
    csrc = os.path.join(os.path.dirname(os.path.abspath(__file__)), "paper_1808_05066_gb300", "csrc")
    h = hashlib.sha256()
    for name in KERNEL_SOURCES:
        with open(os.path.join(csrc, name), "rb") as f:
            h.update(name.encode() + b"\0" + f.read())
    return h.hexdigest()


def ncu_traffic_per_element(kind: str):
    if NCU_TRAFFIC["sources_sha256"] != kernel_sources_digest():
        return None
    return NCU_TRAFFIC["bytes_per_element"].get(kind)


def _dist():
    from paper_1808_05066_gb300.multirank import world
    return world()


def run_reference(args):
    import workloads as wl
    ws, rank, _ = _dist()
    if rank != 0:
        return 0
    spec = dict(wl.WORKLOADS[WORKLOAD])
    n = args.n or spec["n"]
    E = 6 * n ** 3
    rates, cores, desc = oracle_throughput(E, max(1, args.cpu_per_core // 3), steps=args.steps,
                                           warmup=args.warmup, n_override=args.n)
    value = statistics.median(rates)
    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": 1000.0 * E / value, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic", "impl": "reference",
            "config": {"workload": WORKLOAD, "elements": E, "p": 3, "dim": 3, "physics": "navier-stokes",
                       "precision": "fp64", "l2": "per-element working set, host"},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": desc},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


def mixed_degree_leg(args, local, barrier, max_over_ranks, ws):
    """Elements/s of the FP64 assemble + condense of the mixed-degree workload (one persistent
    launch per step over the element classes), with the class census and, on request, one BDF2
    Newton step."""
    import torch
    from paper_1808_05066_gb300 import hdg
    from paper_1808_05066_gb300.workload import DeviceWorkload
    name = "ns3d_mixed_tgv"
    try:
        W = DeviceWorkload(name, device=local, n_override=args.n)
        E = W.info["n_elem"]
        dev = W.dev
        for _ in range(2):
            W.status.zero_()
            W.assemble(hdg.HDG_PREC_FP64)
        torch.cuda.synchronize(dev)
        hdg.hdg_profile_reset(W.ctx.handle)
        barrier()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(args.mixed_degree_steps):
            W.assemble(hdg.HDG_PREC_FP64)
        b.record()
        torch.cuda.synchronize(dev)
        ms = max_over_ranks(a.elapsed_time(b))
        launches, _ = hdg.hdg_profile_read(W.ctx.handle, hdg.HDG_KERNEL_PCLASS)
        bad = int((W.status != 0).sum())
        census = {int(p): int((W.p_elem == p).sum()) for p in (1, 2, 3, 4)}
        out = {"workload": name, "elements": E, "degrees": census,
               "face_degree": "max(p_L, p_R)", "value": ws * E * args.mixed_degree_steps / (ms / 1000.0),
               "unit": "elem/s", "ms_per_step": ms / args.mixed_degree_steps, "steps": args.mixed_degree_steps,
               "precision": "fp64", "launches_per_step": launches / args.mixed_degree_steps,
               "elements_flagged": bad,
               "bytes_written_per_step": 8 * (W.info["len_S"] + W.info["len_g"] + W.info["len_recov"] +
                                              W.info["len_R"])}
        # the FP64 pipe roofline of the fused launch: the flops of every element's class and size
        from paper_1808_05066_gb300.workload import FP64_PIPE_TFLOPS, class_flops_per_element
        lay = W.mesh.layout()
        import numpy as _np
        tdeg = _np.zeros(E, dtype=_np.int64)
        face_of, _, _ = W.mesh.topology()
        tdeg = lay["face_deg"][face_of].max(axis=1)
        ntq = _np.diff(lay["toff"])
        flops = sum(class_flops_per_element(int(pk), int(pt), int(nt))
                    for pk, pt, nt in zip(W.p_elem, tdeg, ntq))
        tf = flops * args.mixed_degree_steps / (ms / 1000.0) / 1e12
        out["roofline"] = {"bound": "fp64", "achieved": tf, "peak": FP64_PIPE_TFLOPS, "unit": "TFLOP/s",
                           "frac": tf / FP64_PIPE_TFLOPS, "kernel": "k_pclass_fused",
                           "peak_source": "derived: 152 SMs x 2 FP64 FMA/clk x 2.07 GHz (a DFMA probe measured 1.20)",
                           "flops_per_step": flops}
        if args.mixed_degree_newton:
            del W.S, W.recov
            torch.cuda.empty_cache()
            hdg.hdg_ctx_set_trace_solver(W.ctx.handle, hdg.HDG_SOLVER_GMRES, 1e-12, 600)
            Vn, Vhn = W.V.clone(), W.Vhat.clone()
            barrier()
            t0 = time.perf_counter()
            it, rn, rh, tr = hdg.hdg_newton_step(W.ctx.handle, Vn, Vhn, W.V, W.V, W.dt, 2, hdg.HDG_PREC_FP64, 1e-10,
                                                 8, history=True)
            torch.cuda.synchronize(dev)
            out["newton_step"] = {"wall_ms": 1e3 * (time.perf_counter() - t0), "newton_updates": it,
                                  "final_res_norm": rn, "residual_history": rh, "trace_iterations": tr}
        W.close()
        return out
    except Exception as exc:  # recorded, not hidden
        return {"error": str(exc)}


def main():
    args = parse()
    if args.impl == "reference":
        return run_reference(args)
    ws, rank, local = _dist()
    import torch
    import torch.distributed as dist

    from paper_1808_05066_gb300 import hdg
    from paper_1808_05066_gb300.workload import (DeviceWorkload, algorithmic_bytes_per_element, flops_per_element,
                                                 method_flops_per_element, slice_flops_per_element)
    if ws > 1:
        dist.init_process_group("nccl", init_method="env://")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    W = DeviceWorkload(WORKLOAD, device=local, n_override=args.n)
    E = W.n_elem
    prec = hdg.HDG_PREC_MIXED if args.precision == "mixed" else hdg.HDG_PREC_FP64
    stream = torch.cuda.current_stream(dev)

    def barrier():
        if ws > 1:
            dist.barrier()
        torch.cuda.synchronize(dev)

    from paper_1808_05066_gb300.multirank import max_over_ranks as _mor

    def max_over_ranks(x):
        return _mor(x, device=dev)

    for _ in range(args.warmup):
        W.assemble(prec)
    torch.cuda.synchronize(dev)
    if int(W.status.abs().sum()) != 0:
        raise RuntimeError("element status flags set during warm-up")
    # ---------------- device-resident timing
    hdg.hdg_profile_reset(W.ctx.handle)
    hdg.hdg_profile_enable(W.ctx.handle, True)
    gpu_index = int(os.environ.get("CUDA_VISIBLE_DEVICES", str(local)).split(",")[0]) if \
        os.environ.get("CUDA_VISIBLE_DEVICES", "").split(",")[0].isdigit() else local
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with ClockSampler(gpu_index) as clk:
        barrier()
        ev0.record(stream)
        for _ in range(args.steps):
            W.assemble(prec)
        ev1.record(stream)
        barrier()
    ms = ev0.elapsed_time(ev1)
    ms = max_over_ranks(ms)
    ms_per_step = ms / args.steps
    value = ws * E * args.steps / (ms / 1000.0)
    classes = {"pointwise": hdg.HDG_KERNEL_POINTWISE, "assemble": hdg.HDG_KERNEL_ASSEMBLE,
               "condense": hdg.HDG_KERNEL_CONDENSE, "mixed_operators": hdg.HDG_KERNEL_MIXED_OPERATORS,
               "mixed_assemble": hdg.HDG_KERNEL_MIXED_ASSEMBLE,
               "mixed_prep": hdg.HDG_KERNEL_MIXED_PREP, "mixed_condense": hdg.HDG_KERNEL_MIXED_CONDENSE}
    prof = {k: hdg.hdg_profile_read(W.ctx.handle, c) for k, c in classes.items()}
    launches_total, _ = hdg.hdg_profile_read(W.ctx.handle, -1)
    hdg.hdg_profile_enable(W.ctx.handle, False)
    dom = max((k for k in prof if prof[k][0] > 0), key=lambda k: prof[k][1])
    dom_launches, dom_ms = prof[dom]
    viscous = W.spec["reynolds"] > 0
    clocks = clk.summary()
    sm_max = clocks.get("sm_max_mhz") or 2070.0
    if dom in ("assemble", "condense"):
        work = flops_per_element(W.info, viscous, dom) * E * args.steps
        # FP64 DFMA pipe: 152 SMs x 2 DFMA/clk x 2 flop x max SM clock
        peak = 152 * 4 * sm_max * 1e6 / 1e12
        roof = {"bound": "alu", "achieved": work / (dom_ms / 1e3) / 1e12, "peak": peak, "unit": "TFLOP/s",
                "peak_source": "derived: 152 SMs x 2 FP64 FMA/clk x max SM clock", "kernel": dom,
                "launches": dom_launches, "avg_launch_ms": dom_ms / max(dom_launches, 1), "traffic": None}
    else:
        # mixed form: the dominant kernel against HBM with the method's algorithmic bytes (for
        # the condensation the S, X, y, g it writes) and against the measured sustained bf16
        # rate with the method's own flops (the kernel runs inside a long step); whichever
        # fraction is larger names the bound. The exact-slice products the tensor cores execute
        # to reach FP64 accuracy are reported beside it (slice_products), not as useful work.
        pk = measured_peaks()
        kind = dom if dom in ("mixed_assemble", "mixed_condense") else "mixed_condense"
        dom_ms_k = prof[kind][1]
        secs = dom_ms_k / 1e3
        method = method_flops_per_element(W.info, viscous, kind) * E * args.steps / secs / 1e12
        slices = slice_flops_per_element(W.info, viscous, kind) * E * args.steps / secs / 1e12
        bpe = algorithmic_bytes_per_element(W.info, viscous, kind)
        hbm = bpe * E * args.steps / secs / 1e9
        launches_k = max(prof[kind][0], 1)
        tpe = ncu_traffic_per_element(kind)
        roof = {"bound": "hbm", "achieved": hbm, "peak": pk["hbm"], "unit": "GB/s", "peak_source": pk["hbm_source"],
                "kernel": kind, "launches": prof[kind][0], "avg_launch_ms": dom_ms_k / launches_k,
                "bytes_per_element": bpe,
                "traffic": None if tpe is None else tpe * E * args.steps / launches_k,
                "traffic_source": NCU_TRAFFIC["source"] if tpe is not None else "kernel sources changed since the capture",
                "tensor": {"achieved": method, "peak": pk["bf16"], "unit": "TFLOP/s", "frac": method / pk["bf16"],
                           "peak_source": pk["bf16_source"], "work": "the method's own flops (FP64-form count)"},
                "slice_products": {"achieved": slices, "unit": "TFLOP/s", "frac_of_bf16_peak": slices / pk["bf16"],
                                   "work": "useful bf16 exact-slice product flops (21 per FP64-accurate product)"}}
        if method / pk["bf16"] > hbm / pk["hbm"]:
            roof["bound"] = "tensor"
            roof["achieved"], roof["peak"], roof["unit"] = method, pk["bf16"], "TFLOP/s"
            roof["peak_source"] = pk["bf16_source"]
    if roof.get("achieved") is not None:
        roof["frac"] = roof["achieved"] / roof["peak"]
    shares = {k: (prof[k][1] / sum(v[1] for v in prof.values()) if prof[k][1] else 0.0) for k in prof}

    # ---------------- the same call replayed as a CUDA graph (hdg_assemble_condense_graph): the
    # first call captures, the timed ones replay; the difference to the ordinary call is the
    # host launch work the graph saves
    graph_replay = None
    try:
        def graph_call():
            hdg.hdg_assemble_condense_graph(W.ctx.handle, W.V, W.Vhat, W.hist, W.mass_coef, prec, W.S, W.g,
                                            W.recov, W.R, W.status)
        graph_call()
        torch.cuda.synchronize(dev)
        r0 = hdg.hdg_ctx_graph_replays(W.ctx.handle)
        ga, gb = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ga.record()
        for _ in range(args.steps):
            graph_call()
        gb.record()
        torch.cuda.synchronize(dev)
        gms = ga.elapsed_time(gb) / args.steps
        graph_replay = {"ms_per_step": gms, "value": E / (gms / 1000.0), "unit": UNIT,
                        "replays": hdg.hdg_ctx_graph_replays(W.ctx.handle) - r0,
                        "ordinary_ms_per_step": ms_per_step}
    except Exception as exc:  # recorded, not hidden
        graph_replay = {"error": str(exc)}

    # ---------------- the plain FP64 GPU form on the same workload, and the accuracy of
    # the headline form against it on every element (relative Frobenius norm of S)
    fp64_form = None
    if prec != hdg.HDG_PREC_FP64 and args.fp64_steps > 0:
        S_head = W.S.clone() if W.S.numel() * 8 < 0.3 * torch.cuda.get_device_properties(dev).total_memory else None
        W.assemble(hdg.HDG_PREC_FP64)
        barrier()
        ev0.record(stream)
        for _ in range(args.fp64_steps):
            W.assemble(hdg.HDG_PREC_FP64)
        ev1.record(stream)
        barrier()
        ms64 = max_over_ranks(ev0.elapsed_time(ev1))
        fp64_form = {"value": ws * E * args.fp64_steps / (ms64 / 1000.0), "unit": UNIT,
                     "ms_per_step": ms64 / args.fp64_steps, "steps": args.fp64_steps}
        if S_head is not None:
            err = 0.0
            for e0 in range(0, E, 4096):
                d = (S_head[e0:e0 + 4096] - W.S[e0:e0 + 4096]).flatten(1).norm(dim=1)
                n = W.S[e0:e0 + 4096].flatten(1).norm(dim=1)
                err = max(err, float((d / n).max()))
            fp64_form["max_rel_err_S_vs_fp64"] = err
            del S_head
        fp64_form["speedup_of_headline"] = value / fp64_form["value"]

    # ---------------- end to end through the C-ABI with host buffers
    e2e = None
    if not args.no_e2e:
        pin = dict(pin_memory=True)
        hV = W.V.cpu().pin_memory()
        hVh = W.Vhat.cpu().pin_memory()
        hS = torch.empty(W.S.shape, dtype=torch.float64, **pin)
        hg = torch.empty(W.g.shape, dtype=torch.float64, **pin)
        dV = torch.empty_like(W.V)
        dVh = torch.empty_like(W.Vhat)
        h2d = hV.numel() * 8 + hVh.numel() * 8
        d2h = hS.numel() * 8 + hg.numel() * 8

        def e2e_step():
            # inputs from pinned host memory; S and g back to pinned host memory through the
            # public entry point that overlaps each chunk's copy with the next chunk's kernels
            dV.copy_(hV, non_blocking=True)
            dVh.copy_(hVh, non_blocking=True)
            W.assemble_to_host(hS, hg, prec, V=dV, Vhat=dVh)

        for _ in range(max(1, min(args.warmup, 2))):
            e2e_step()
        barrier()
        ev0.record(stream)
        for _ in range(args.steps):
            e2e_step()
        ev1.record(stream)
        barrier()
        ms2 = max_over_ranks(ev0.elapsed_time(ev1))
        e2e = {"value": ws * E * args.steps / (ms2 / 1000.0), "unit": UNIT, "h2d_bytes_per_step": h2d,
               "d2h_bytes_per_step": d2h}
        del hS, hg

    # ---------------- one implicit BDF2 Newton step (assemble+condense, GMRES trace
    # solve, recovery, update, residual norms) to |R| <= 1e-10 max(1, |R0|)
    def newton_step(p, rtol=1e-12):
        """One BDF2 step (u^{n-1} = u^n) through hdg_newton_step; the first call sizes the
        workspaces, the second is timed. rtol 0: inexact Newton (Eisenstat-Walker forcing)."""
        try:
            hdg.hdg_ctx_set_trace_solver(W.ctx.handle, hdg.HDG_SOLVER_AUTO, rtol, 600)
            for timed in (False, True):
                Vn, Vhn = W.V.clone(), W.Vhat.clone()
                barrier()
                t0 = time.perf_counter()
                it, rn, rh, tr = hdg.hdg_newton_step(W.ctx.handle, Vn, Vhn, W.V, W.V, W.dt, 2, p, 1e-10, 8,
                                                     history=True)
                torch.cuda.synchronize(dev)
                wall = 1e3 * (time.perf_counter() - t0)
                del Vn, Vhn
            hdg.hdg_ctx_set_trace_solver(W.ctx.handle)
            return {"wall_ms": wall, "newton_updates": it, "final_res_norm": rn, "tol": 1e-10,
                    "trace_iterations": tr, "residual_history": rh,
                    "trace_solver": "GMRES(30), face-block Jacobi, " +
                                    ("rtol %g" % rtol if rtol > 0 else "Eisenstat-Walker forcing (inexact Newton)")}
        except Exception as exc:  # recorded, not hidden
            return {"error": str(exc)}

    newton = newton64 = newton_ew = None
    if not args.no_newton:
        newton = newton_step(prec)
        newton_ew = newton_step(prec, 0.0)
        if prec != hdg.HDG_PREC_FP64:
            newton64 = newton_step(hdg.HDG_PREC_FP64)

    # ---------------- mixed-degree batch: the 32^3 cube (196,608 tets) with degrees 1..4 drawn per
    # element, FP64, every element in one persistent fused launch per step
    mixed_degree = None
    cube_n = W.spec["n"]
    if not args.no_mixed_degree:
        W.close()
        del W
        torch.cuda.empty_cache()
        mixed_degree = mixed_degree_leg(args, local, barrier, max_over_ranks, ws)

    # ---------------- CPU baseline (oracle), rank 0 at N=1 only
    cpu = None
    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        rates, cores, desc = oracle_throughput(E, args.cpu_per_core, steps=2, warmup=0, n_override=args.n)
        cpu = {"value": max(rates), "unit": UNIT, "cores": cores, "kind": "oracle",
               "sample": desc + "; best of 2 passes over the same sample"}

    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_per_step, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None,
            "dtype": "bf16x6-slice(FP64-accurate)+f32+f64" if prec == hdg.HDG_PREC_MIXED else "f64",
            "data": "synthetic",
            "config": {"workload": WORKLOAD, "elements_per_gpu": E, "dim": 3, "p": 3, "physics": "navier-stokes",
                       "mesh": f"{cube_n}^3 periodic cube x 6 tets", "precision": args.precision,
                       "l2": "inputs+outputs larger than L2 (S alone 26.5 GB written per step)",
                       "parallelism": f"replica per GPU x{ws}"},
            "roofline": roof, "kernel_time_share": shares, "gpu_launches": launches_total,
            "fp64_form": fp64_form, "graph_replay": graph_replay, "newton_step": newton, "newton_step_inexact": newton_ew,
            "newton_step_fp64": newton64, "mixed_degree": mixed_degree,
            "clocks": clocks, "e2e": e2e, "cpu_baseline": cpu,
        }
        print(json.dumps(line), flush=True)
    if ws > 1:
        dist.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
