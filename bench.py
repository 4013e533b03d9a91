#!/usr/bin/env python
"""Throughput benchmark of the superiorized hyperslab-projection path on GB300.

A step is one superiorized solve of the CT 512x512 configuration (360 angles x
725 bins, Siddon CSR, FP32 values, int32 indices): the iterate reset to
box(0), then 200 iterations of Algorithm 1 (TV perturbation phase followed by
one Cimmino sweep with the fused proximity and stopping bookkeeping).  The
headline value is nnz * sweeps / s with A resident in HBM (the sweep strategy
and its launch shapes chosen by the library's tuner at create); the e2e value
is the same metric through the C ABI with host buffers (new bounds and x0 in,
x out, copies inside the timed region).  The roofline is that of the whole
sweep (every launch of one application of T) against the algorithmic bytes
of a sweep.  Extra variants (block-iterative, BF16 values, batched seismic,
radiotherapy, tiny CT) are reported under "variants", the error of 16-bit
values against the FP64 oracle on the original A under "precision", and the
serving mix under "serving".

Usage: python bench.py [--gpus N --steps K --warmup W] [--impl reference]
Under torchrun each rank runs an independent replica (weak scaling).
"""
from __future__ import annotations

import argparse
import dataclasses
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

METRIC = "nnz·sweeps/s"
UNIT = "nnz*sweeps/s"
CT512 = dict(N=512, nang=360, nbin=725, I0=5e3, delta=0.02, seed_phantom=201, seed_noise=202)
SUP = dict(gamma=0.5, alpha=0.99, n_red=1)
SWEEPS = 200          # iterations of one CT 512x512 solve (the configuration's count)


def log(*a):
    print(*a, file=sys.stderr, flush=True)


def dist_env():
    return (int(os.environ.get("RANK", 0)), int(os.environ.get("WORLD_SIZE", 1)),
            int(os.environ.get("LOCAL_RANK", 0)))


def ct512():
    import synth
    return synth.ct_problem(**CT512)


# ------------------------------------------------------------------ clocks --

class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons during a region."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_id: str):
        self.gpu = gpu_id
        self.lines = []
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "100",
                                          "-i", self.gpu], stdout=subprocess.PIPE,
                                         stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except Exception:
            self.proc = None

    def _read(self):
        for ln in self.proc.stdout:
            self.lines.append(ln.strip())

    def stop(self):
        if not self.proc:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.t.join(timeout=2)
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                smax.append(float(f[2]))
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(smax) if smax else None,
                "samples": len(sm), "reasons": sorted(reasons)}


def gpu_id_for(dev: int) -> str:
    import torch
    try:
        u = str(torch.cuda.get_device_properties(dev).uuid)
        return u if u.startswith("GPU-") else "GPU-" + u
    except Exception:
        vis = os.environ.get("CUDA_VISIBLE_DEVICES", "")
        ids = [v for v in vis.split(",") if v.strip()]
        return ids[dev] if dev < len(ids) else str(dev)


def peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


# ------------------------------------------------------------ CPU baseline --

_ORACLE = {}   # the oracle's setup of the CT 512x512 workload, shared with forked workers


def _oracle_setup(prob):
    import oracle as O
    if "S" not in _ORACLE:
        S, l, u, lo, hi = O.from_problem(prob)
        _ORACLE.update(S=S, l=l, u=u, lo=lo, hi=hi,
                       ob=O.Objective(O.OBJ_TV_ISO, prob.shape), n=prob.A.n)
    return _ORACLE


def _oracle_iterations(seconds: float, seed: int = 0):
    """Superiorized Cimmino iterations of the oracle (as it stands) from box(0)
    until `seconds` pass; returns (iterations, elapsed s)."""
    import oracle as O
    d = _ORACLE
    P = O.Params(**SUP)
    st = O.PertState()
    x = np.zeros(d["n"])
    it = 0
    t0 = time.perf_counter()
    while True:
        x, _, _ = O.perturbation_phase(d["ob"], x, st, P)
        x, _ = O.sweep(d["S"], O.CIMMINO, d["l"], d["u"], 1.0, d["lo"], d["hi"], x)
        it += 1
        el = time.perf_counter() - t0
        if el >= seconds:
            return it, el


def cpu_baselines(prob, seconds: float):
    """The FP64 oracle timed on this host's cores on a bounded sample of the
    headline workload: one process (one thread: scipy's sparse products are
    single-threaded), then one process per core, each running the same
    iterations (the aggregate rate of replicas; the setup is built once and
    shared by the forked workers).  Must run before the first CUDA call (the
    workers are forked)."""
    import multiprocessing as mp
    nnz = prob.A.nnz
    _oracle_setup(prob)
    it1, el1 = _oracle_iterations(seconds)
    cores = os.cpu_count() or 1
    ctx = mp.get_context("fork")
    with ctx.Pool(cores) as pool:
        res = pool.map(_oracle_iterations, [seconds] * cores)
    its = sum(r[0] for r in res)
    el = max(r[1] for r in res)
    single = {"value": nnz * it1 / el1, "unit": UNIT, "cores": 1, "kind": "oracle",
              "sample": f"{it1} superiorized Cimmino iterations of the CT 512x512 workload from "
                        f"box(0) ({el1:.1f} s, FP64 numpy/scipy oracle, one process)"}
    allc = {"value": nnz * its / el, "unit": UNIT, "cores": cores, "kind": "oracle",
            "sample": f"{cores} processes (one per host core) each running superiorized Cimmino "
                      f"iterations of the CT 512x512 workload from box(0) for {seconds:.0f} s "
                      f"({its} iterations in all, FP64 numpy/scipy oracle)",
            "single_thread": single}
    return allc


def reference_arm(args):
    """The reference arm: the FP64 oracle (there is no installable reference
    implementation), on this host's cores, on a bounded sample of the same
    workload and metric (each step a few superiorized iterations)."""
    rank, world, _ = dist_env()
    if rank != 0:
        return 0
    prob = ct512()
    nnz = prob.A.nnz
    import oracle as O
    d = _oracle_setup(prob)
    P = O.Params(**SUP)
    st = O.PertState()
    x = np.zeros(prob.A.n)
    per_step = 2   # iterations per step: a bounded sample of a 200-iteration solve

    def step(x):
        for _ in range(per_step):
            x, _, _ = O.perturbation_phase(d["ob"], x, st, P)
            x, _ = O.sweep(d["S"], O.CIMMINO, d["l"], d["u"], 1.0, d["lo"], d["hi"], x)
        return x

    for _ in range(args.warmup):
        x = step(x)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        x = step(x)
    el = time.perf_counter() - t0
    v = nnz * per_step * args.steps / el
    sample = (f"{args.steps} steps of {per_step} superiorized Cimmino iterations (TV perturbation "
              f"+ sweep) of the CT 512x512 workload, FP64 numpy/scipy oracle, one process")
    out = {"impl": "reference", "metric": METRIC, "value": v, "unit": UNIT, "n_gpus": world,
           "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * el / args.steps,
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
           "data": "synthetic", "config": config_of(prob),
           "cpu_baseline": {"value": v, "unit": UNIT, "cores": 1, "kind": "oracle",
                            "sample": sample},
           "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(out), flush=True)
    return 0


def config_of(prob):
    return {"workload": "ct512_cimmino_tv_f32", "image": "512x512", "angles": 360, "bins": 725,
            "m": prob.A.m, "n": prob.A.n, "nnz": prob.A.nnz, "I0": 5e3, "slab_delta": 0.02,
            "perturbation": "TV, beta=0.5*0.99^l, n_red=1", "relaxation": 1.0,
            "step": f"one solve: x <- box(0), then {SWEEPS} superiorized Cimmino iterations",
            "l2": "inputs larger than L2 (A values+indices ~0.96 GB > 126 MB L2)"}


# ------------------------------------------------------------------ ours ----

def time_iterations(ctx, pk, K, W, params_kw, with_timing=True):
    """Run W untimed iterations, then K timed ones in one suppy_run call;
    returns (elapsed ms, {kind: (kernel ms, launches)}, library launches)."""
    import torch
    s = torch.cuda.current_stream()
    if W:
        ctx.suppy_run(pk.suppy_params_default(max_sweeps=W, **params_kw))
    torch.cuda.synchronize()
    if with_timing:
        ctx.suppy_timing_enable(True)
    l0 = ctx.suppy_launch_count()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(s)
    ctx.suppy_run(pk.suppy_params_default(max_sweeps=K, **params_kw))
    e1.record(s)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    nl = ctx.suppy_launch_count() - l0
    kt = {k: ctx.suppy_kernel_time(k) for k in (0, 1, 2, 3)} if with_timing else {}
    if with_timing:
        ctx.suppy_timing_enable(False)
    return ms, kt, nl


KIND = {0: "row pass", 1: "column pass / finalize", 2: "perturbation", 3: "split (CQ) step"}
STRATEGY = {1: "one pass (L2-reduction scatter)", 2: "two passes (CSR row pass, CSC column pass)",
            3: "tiled one pass"}


def kind_name(strategy, k):
    if strategy == 3 and k == 0:
        return "tiled sweep"
    return KIND[k]


def sweep_traffic_from(table, info):
    """DRAM bytes per sweep (all of the sweep's launches) of a capture table
    for this run's strategy and launch shape, or None with the reason.  A
    strategy's entry is one capture or a list of captures of several shapes."""
    ent = table.get(f"ct512_sweep_strategy{info['strategy']}")
    if not ent:
        return None, "no committed capture of this strategy"
    for e in (ent if isinstance(ent, list) else [ent]):
        shape = e.get("shape", {})
        if {k: info.get(k) for k in shape} == shape:
            return float(e["bytes_per_sweep"]), e.get("note")
    return None, "the committed capture is of another launch shape"


def sweep_traffic(info):
    """The committed ncu capture's DRAM bytes per sweep (profiles/traffic.json)
    when it was taken on this run's strategy and launch shape."""
    path = os.path.join(ROOT, "profiles", "traffic.json")
    if not os.path.exists(path):
        return None, "no committed capture"
    try:
        table = json.load(open(path))
    except (OSError, ValueError):
        return None, "unreadable capture table"
    return sweep_traffic_from(table, info)


def sweep_alg_bytes(m, n, nnz, vbytes, B=1):
    """Algorithmic bytes of one application of T (the per-unit figures of the
    measurement plan): A's values and column indices once, per row its
    offset, l, u and weight (16 B), per unknown x read and written and the
    correction (16 B)."""
    return nnz * (vbytes + 4) + m * 16 + n * 16 * B


def kernel_alg_bytes(strategy, kind, m, n, nnz, vb, B=1):
    """Algorithmic bytes a kernel of the sweep carries (its share of one
    sweep's): the pass that reads A carries A's bytes; a second read of A (the
    column pass of the two-pass sweep reads the CSC copy) is traffic, not
    algorithmic bytes.  Row pass: A, the per-row data (16 B); two passes add
    the coefficients written (4 B a row).  Column pass: x read and written,
    coefficients read; finalize: x and the correction read and written.  The
    tiled sweep is the whole sweep."""
    if strategy == 3:
        return sweep_alg_bytes(m, n, nnz, vb, B) if kind == 0 else 0
    if kind == 0:
        return nnz * (vb + 4) + m * 16 * B + (m * 4 * B if strategy == 2 else 0)
    if kind == 1:
        return n * 8 * B + m * 4 * B if strategy == 2 else n * 16 * B
    return 0


def summarize(ctx, prob, K, kt, vb, B=1):
    """Per-kernel times per sweep and the sweep time (the kernels of one
    application of T: kinds 0 and 1)."""
    info = ctx.suppy_info_get()
    strat = info["strategy"]
    A = prob.A
    per = {}
    for k, (tms, nl) in kt.items():
        if nl == 0:
            continue
        if k == 3:
            Aq = prob.meta["split"]["Aq"]
            alg = 2 * Aq.nnz * 8 + (Aq.m + A.n) * 8 + Aq.m * 4 + A.n * 8
        else:
            alg = kernel_alg_bytes(strat, k, A.m, A.n, A.nnz, vb, B)
        ms = tms / K
        per[kind_name(strat, k)] = {"ms_per_sweep": ms, "launches_per_sweep": nl / K,
                                    "alg_bytes_per_sweep": alg,
                                    "gbs_alg": alg / (ms * 1e-3) / 1e9 if alg else None}
    t_sweep = sum(kt[k][0] for k in (0, 1) if k in kt) / K
    tot = sum(kt[k][0] for k in kt) / K
    for k, v in per.items():
        v["share_of_step_kernels"] = v["ms_per_sweep"] / tot if tot else None
    return info, per, t_sweep


def variants(pk, K, W):
    """Secondary workloads (outside the headline timed region)."""
    import torch
    import synth
    out = {}
    Kv = max(20, min(K, 200))

    def run_one(name, prob, metric_units, **kw):
        obj = kw.pop("obj")
        dtype = kw.pop("dtype", pk.SUPPY_F32)
        mode = kw.pop("mode", pk.SUPPY_CIMMINO)
        pkw = kw.pop("params")
        split = kw.pop("split", False)
        B = 1 if prob.l.ndim == 1 else prob.l.shape[1]
        t0 = time.perf_counter()
        ctx = pk.from_problem(prob, obj=obj, dtype=dtype, mode=mode, **kw)
        nnz_q = 0
        if split:
            sp = prob.meta["split"]
            Aq = sp["Aq"]
            ctx.suppy_set_dvc(Aq.row_ptr, Aq.col, Aq.val, Aq.m, sp["sptr"], sp["dvcs"], 1.0)
            nnz_q = Aq.nnz
        t_create = time.perf_counter() - t0
        ms, _, nl = time_iterations(ctx, pk, Kv, W, pkw, with_timing=False)
        _, kt, _ = time_iterations(ctx, pk, Kv, 0, pkw, with_timing=True)
        vb = 4 if dtype == pk.SUPPY_F32 else 2
        info, per, t_sweep = summarize(ctx, prob, Kv, kt, vb, B)
        nnz = prob.A.nnz
        alg = sweep_alg_bytes(prob.A.m, prob.A.n, nnz, vb, B)
        peak, _ = peaks()
        # a split iteration also passes over the dose rows A_q: their entries count
        out[name] = {"value": (nnz + nnz_q) * B * Kv / (ms * 1e-3), "unit": metric_units,
                     "ms_per_step": ms / Kv, "sweep_ms": t_sweep,
                     "sweep_gbs_alg": alg / (t_sweep * 1e-3) / 1e9 if t_sweep else None,
                     "sweep_frac_of_peak": alg / (t_sweep * 1e-3) / 1e9 / peak if t_sweep else None,
                     "m": prob.A.m, "n": prob.A.n, "nnz": nnz, "nrhs": B, "kernels": per,
                     "create_s": t_create, "strategy": info["strategy"],
                     "scatter": info["scatter"], "nblocks": info["nblocks"], "tma": info["tma"],
                     "transposed_rows": info["transposed_rows"],
                     "scatter_patch": info["scatter_patch"], "a_dtype": info["a_dtype"],
                     "launches_per_step": nl / Kv}
        if info["strategy"] == 3:
            out[name]["tiles"] = {k: info[k] for k in ("tiles", "chunks", "tile_warps1",
                                                       "tile_warps2", "tile_coef_warps",
                                                       "tile_ring", "tile_stream_bytes",
                                                       "tile_segments")}
        if split:
            out[name]["nnz_split"] = nnz_q
        ctx.close()
        torch.cuda.synchronize()

    prob = ct512()
    for strat, tag in ((pk.STRATEGY_TILED, "tiled"), (pk.STRATEGY_TWO_PASS, "twopass"),
                       (pk.STRATEGY_ONE_PASS, "onepass")):
        run_one(f"ct512_cimmino_tv_f32_{tag}", prob, UNIT, obj=pk.SUPPY_OBJ_TV_ISO, params=SUP,
                strategy=strat, tune=1)
    run_one("ct512_cimmino_tv_f32_twopass_notma", prob, UNIT, obj=pk.SUPPY_OBJ_TV_ISO, params=SUP,
            strategy=pk.STRATEGY_TWO_PASS, tma=-1)
    run_one("ct512_emr_tv_f32", prob, UNIT, obj=pk.SUPPY_OBJ_TV_ISO, mode=pk.SUPPY_EMR,
            params=SUP, tune=1)
    run_one("ct512_el_tv_f32", prob, UNIT, obj=pk.SUPPY_OBJ_TV_ISO, mode=pk.SUPPY_EL,
            params=SUP, tune=1)
    run_one("ct512_drop_tv_f32", prob, UNIT, obj=pk.SUPPY_OBJ_TV_ISO, mode=pk.SUPPY_DROP,
            params=SUP, tune=1)
    run_one("ct512_cimmino_tv_bf16", prob, UNIT, obj=pk.SUPPY_OBJ_TV_ISO, dtype=pk.SUPPY_BF16,
            params=SUP, tune=1)
    run_one("ct512_cimmino_tv_f16", prob, UNIT, obj=pk.SUPPY_OBJ_TV_ISO, dtype=pk.SUPPY_F16,
            params=SUP, tune=1)
    prob.blocks = synth.angle_blocks(360, 725, 36)
    run_one("ct512_bip36_tv_f32", prob, UNIT, obj=pk.SUPPY_OBJ_TV_ISO, mode=pk.SUPPY_BIP,
            params=SUP, tune=1)
    run_one("ct512_bip36_tv_f32_twopass", prob, UNIT, obj=pk.SUPPY_OBJ_TV_ISO, mode=pk.SUPPY_BIP,
            params=SUP, strategy=pk.STRATEGY_TWO_PASS, tune=1)
    del prob
    seis = synth.seismic_problem(nrhs=16)
    run_one("seismic_b16_atv_f32", seis, "nnz*rhs*sweeps/s", obj=pk.SUPPY_OBJ_TV_ANISO,
            params=SUP)
    run_one("seismic_b16_atv_f32_onepass", seis, "nnz*rhs*sweeps/s", obj=pk.SUPPY_OBJ_TV_ANISO,
            params=SUP, strategy=pk.STRATEGY_ONE_PASS)
    run_one("seismic_b16_atv_drop_f32", seis, "nnz*rhs*sweeps/s", obj=pk.SUPPY_OBJ_TV_ANISO,
            mode=pk.SUPPY_DROP, params=SUP)
    seis.l, seis.u = seis.l[:, 0].copy(), seis.u[:, 0].copy()
    run_one("seismic_b1_atv_f32", seis, UNIT, obj=pk.SUPPY_OBJ_TV_ANISO, params=SUP, tune=1)
    del seis
    rt = synth.rt_problem()
    run_one("rt_bip3_meandose_f32", rt, UNIT, obj=pk.SUPPY_OBJ_LINEAR, mode=pk.SUPPY_BIP,
            params=dict(gamma=1.0, alpha=0.99, n_red=1))
    del rt
    # the horseshoe plan as a split problem: DVCs by the CQ step, slabs by EMR
    # (the paper's choice for the linear constraints), restarts every 500
    rts = synth.rt_split_problem()
    run_one("rt_split_dvc_emr_meandose_f32", rts, UNIT, obj=pk.SUPPY_OBJ_LINEAR,
            mode=pk.SUPPY_EMR, params=dict(gamma=1.0, alpha=0.7, n_red=1, restart_every=500),
            split=True)
    del rts
    tiny = synth.ct_problem()
    run_one("ct64_cimmino_tv_f32", tiny, UNIT, obj=pk.SUPPY_OBJ_TV_ISO, params=SUP)
    return out


def precision(pk):
    """Error of 16-bit storage of A's values against the FP64 oracle on the
    original (FP32) values, and the parity gate against the oracle on the
    rounded values.  CT 64x64 (configuration 1): the full 100-iteration
    superiorized run from box(0).  CT 512x512: one sweep from a seeded point,
    and three superiorized iterations from box(0)."""
    import torch
    import oracle as O
    import synth

    def rounded(v, dt):
        t = torch.from_numpy(np.ascontiguousarray(v, np.float32))
        return (t.to(torch.bfloat16) if dt == pk.SUPPY_BF16 else t.to(torch.float16)).to(
            torch.float32).numpy()

    def rel_l2(a, b):
        a = np.asarray(a, np.float64)
        b = np.asarray(b, np.float64)
        return float(np.linalg.norm(a - b) / np.linalg.norm(b))

    def rel(a, b):
        return float(abs(a - b) / max(abs(b), 1e-300))

    out = {}
    ob_kind = O.OBJ_TV_ISO
    for label, prob, K in (("ct64_100_iterations", synth.ct_problem(), 100),
                           ("ct512_3_iterations", ct512(), 3)):
        ob = O.Objective(ob_kind, prob.shape)
        P = O.Params(max_sweeps=K, **SUP)
        S, l, u, lo, hi = O.from_problem(prob)
        r64 = O.run(S, O.CIMMINO, l, u, lo, hi, ob, P)
        sweep64 = None
        if K == 3:
            x0 = np.random.default_rng(7).uniform(0, 1, prob.A.n).astype(np.float32)
            sweep64, _ = O.sweep(S, O.CIMMINO, l, u, 1.0, lo, hi, x0.astype(np.float64))
        for dt, name in ((pk.SUPPY_BF16, "bf16"), (pk.SUPPY_F16, "f16"), (pk.SUPPY_F32, "f32")):
            vals = prob.A.val if dt == pk.SUPPY_F32 else rounded(prob.A.val, dt)
            Sr, lr, ur, lor, hir = O.from_problem(prob, values=vals)
            rr = O.run(Sr, O.CIMMINO, lr, ur, lor, hir, ob, P) if dt != pk.SUPPY_F32 else r64
            ctx = pk.from_problem(prob, obj=pk.SUPPY_OBJ_TV_ISO, dtype=dt, tune=1 if K == 3 else 0)
            st = ctx.suppy_run(pk.suppy_params_default(max_sweeps=K, **SUP))[0]
            xg = ctx.suppy_get_x()
            ph, fh = ctx.suppy_history()
            e = {"x_rel_l2_vs_fp64_oracle_original_A": rel_l2(xg, r64.x),
                 "x_rel_l2_vs_fp64_oracle_rounded_A": rel_l2(xg, rr.x),
                 "final_proximity_rel_vs_original": rel(ph[-1], r64.prox_hist[-1]),
                 "final_proximity_rel_vs_rounded": rel(ph[-1], rr.prox_hist[-1]),
                 "final_objective_rel_vs_original": rel(fh[-1], r64.obj_hist[-1]),
                 "oracle_rounded_vs_original_x_rel_l2": rel_l2(rr.x, r64.x),
                 "sweeps": st["sweeps"]}
            if sweep64 is not None:
                ctx.suppy_set_x(x0)
                ctx.suppy_sweep(pk.suppy_params_default(), 1)
                x1 = ctx.suppy_get_x()
                sr, _ = O.sweep(Sr, O.CIMMINO, lr, ur, 1.0, lor, hir, x0.astype(np.float64))
                e["one_sweep_x_rel_l2_vs_original"] = rel_l2(x1, sweep64)
                e["one_sweep_x_rel_l2_vs_rounded"] = rel_l2(x1, sr)
            out[f"{label}_{name}"] = e
            ctx.close()
            torch.cuda.synchronize()
    return out


def aggregate_over_ranks(ms: float, units: float, world: int):
    """Whole-job figures of N independent replicas: the elapsed time is the
    maximum over ranks, and the throughput is the units all ranks processed
    (each rank `units`) divided by that time."""
    if world > 1:
        import torch
        import torch.distributed as dist
        t = torch.tensor([ms], dtype=torch.float64)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        ms = float(t.item())
    return ms, units * world / (ms * 1e-3)


# ----------------------------------------------------------------- serving --

SERVE_STOP = dict(use_stopping=1, prox_rel=1e-4, patience=5, prox_abs=1e-6, obj_rel=0.0,
                  max_sweeps=500)


def serving_workload(pk, nreq: int, seed: int = 501):
    """The serving mix: Poisson arrivals at 200 requests/s (seed 501); 60% CT
    slices (128^2 / 256^2 / 512^2 with 90x183 / 180x363 / 360x725 geometries),
    25% seismic (128x256 / 256x512), 15% radiotherapy plans (three plan sizes
    on the 50k-300k voxel x 1k-6k beamlet grid, seed 502, OAR caps varied per
    request).  Every request is one set of slab bounds for a registered
    matrix; CT and seismic requests are independent noise realisations."""
    import synth
    rng = np.random.default_rng(seed)
    t = np.cumsum(rng.exponential(1.0 / 200.0, size=nreq))
    kind = rng.choice(3, size=nreq, p=[0.60, 0.25, 0.15])
    ct_geo = [(128, 90, 183), (256, 180, 363), (512, 360, 725)]
    se_geo = [(128, 256, 64, 256), (256, 512, 128, 512)]
    rt_geo = [dict(nx=50, ny=40, nz=25, ns=12, nzb=9), dict(nx=80, ny=50, nz=38, ns=20, nzb=17),
              dict()]
    sub = np.where(kind == 0, rng.integers(0, 3, nreq),
                   np.where(kind == 1, rng.integers(0, 2, nreq), rng.integers(0, 3, nreq)))
    rng_rt = np.random.default_rng(502)
    mats, reqs = [], []
    for k in range(3):
        for g in range(3 if k != 1 else 2):
            idx = np.where((kind == k) & (sub == g))[0]
            if len(idx) == 0:
                continue
            R = len(idx)
            if k == 0:
                N, na, nb = ct_geo[g]
                prob = synth.ct_problem(N, na, nb, I0=5e3, delta=0.02, seed_phantom=201 + g,
                                        seed_noise=1000 * (g + 1), nrhs=max(R, 2))
                spec = dict(obj=pk.SUPPY_OBJ_TV_ISO, mode=pk.SUPPY_CIMMINO,
                            sup=dict(gamma=0.5, alpha=0.99, n_red=1), name=f"ct{N}")
                cols = [(prob.l[:, j], prob.u[:, j]) for j in range(R)]
            elif k == 1:
                H, W, ns, nr = se_geo[g]
                prob = synth.seismic_problem(H, W, ns, nr, nrhs=max(R, 2),
                                             seed_noise=2000 * (g + 1))
                spec = dict(obj=pk.SUPPY_OBJ_TV_ANISO, mode=pk.SUPPY_CIMMINO,
                            sup=dict(gamma=0.5, alpha=0.99, n_red=1), name=f"seismic{H}x{W}")
                cols = [(prob.l[:, j], prob.u[:, j]) for j in range(R)]
            else:
                prob = synth.rt_problem(**rt_geo[g])
                spec = dict(obj=pk.SUPPY_OBJ_LINEAR, mode=pk.SUPPY_BIP,
                            sup=dict(gamma=1.0, alpha=0.99, n_red=1),
                            name=f"rt{prob.meta['n_body']}x{prob.meta['beamlets']}")
                nt, n1 = prob.meta["n_target"], prob.meta["n_oar1"]
                cols = []
                for _ in range(R):
                    u = prob.u.copy()
                    u[nt:nt + n1] = rng_rt.uniform(15.0, 25.0)
                    u[nt + n1:] = rng_rt.uniform(25.0, 35.0)
                    cols.append((prob.l, u))
            mats.append((prob, spec))
            for j, i in enumerate(idx):
                reqs.append((float(t[i]), len(mats) - 1, cols[j][0], cols[j][1]))
    reqs.sort(key=lambda r: r[0])
    return mats, reqs


def _serve_batched(pk, mats, reqs, dtype):
    """The requests through one continuous-batching server (A stored as dtype);
    returns its figures and per request (final proximity, final objective,
    sweeps)."""
    import torch
    srv = pk.Server(slots=32, check_every=8)
    mids = []
    for prob, spec in mats:
        P = pk.suppy_params_default(**spec["sup"], **SERVE_STOP)
        mids.append(srv.suppy_server_add_matrix(prob, P, dtype=dtype, mode=spec["mode"],
                                                obj=spec["obj"]))
    ids = [None] * len(reqs)
    t0 = srv.suppy_server_clock()
    nxt = 0
    while True:
        now = srv.suppy_server_clock() - t0
        while nxt < len(reqs) and reqs[nxt][0] <= now:
            ids[nxt] = srv.suppy_server_submit(mids[reqs[nxt][1]], reqs[nxt][2], reqs[nxt][3])
            nxt += 1
        r, w = srv.suppy_server_step()
        if nxt == len(reqs) and r == 0 and w == 0:
            break
    lat, queue, service, fin, per = [], [], [], [], []
    for k, rid in enumerate(ids):
        info, _ = srv.suppy_server_query(rid)
        lat.append(info["t_done"] - t0 - reqs[k][0])
        queue.append(info["t_start"] - t0 - reqs[k][0])
        service.append(info["t_done"] - info["t_start"])
        fin.append(info["t_done"] - t0)
        per.append((info["proximity"], info["objective"], info["sweeps"]))
    peak_bytes = srv.suppy_server_device_bytes()
    srv.close()
    torch.cuda.synchronize()
    name = {pk.SUPPY_BF16: "bf16 A", pk.SUPPY_F16: "f16 A", pk.SUPPY_F32: "f32 A"}.get(
        dtype, "16-bit A (FP16 or BF16 per matrix, the smaller rounding error)")
    arrivals = reqs[-1][0]
    figs = {"solves_per_s": len(reqs) / max(fin), "p50_s": float(np.percentile(lat, 50)),
            "p99_s": float(np.percentile(lat, 99)), "makespan_s": max(fin),
            "queue_p50_s": float(np.percentile(queue, 50)),
            "queue_p99_s": float(np.percentile(queue, 99)),
            "service_p50_s": float(np.percentile(service, 50)),
            "service_p99_s": float(np.percentile(service, 99)),
            # the offered load is sustained when completions keep pace with
            # arrivals (throughput at least 95% of the arrival rate)
            "offered_rate_per_s": len(reqs) / max(arrivals, 1e-9),
            "sustains_arrival_rate": bool(len(reqs) / max(fin) >= 0.95 * len(reqs) / max(arrivals, 1e-9)),
            "mean_sweeps": float(np.mean([p[2] for p in per])),
            "dtype": name + ", f32 x, f64 acceptance", "device_bytes_end": int(peak_bytes)}
    return figs, per


def serving(pk, nreq: int):
    """Batched continuous-batching server (16-bit A: FP16 or BF16 per matrix,
    whichever rounds it with the smaller error; and FP32 A for a comparison
    at equal precision) against one-at-a-time FP32 solves of the same requests
    (arrival times kept, queueing included).  Per request, the final
    proximity and objective are compared with the one-at-a-time solve; a
    request that stops at another sweep than its one-at-a-time solve is also
    compared at equal sweep counts (the one-at-a-time history at the batched
    request's last sweep)."""
    import torch
    mats, reqs = serving_workload(pk, nreq)
    batched, per_b = _serve_batched(pk, mats, reqs, pk.SUPPY_HALF_AUTO)
    # the 16-bit format the library takes for each matrix
    fmt = {}
    for prob, spec in mats:
        one = dataclasses.replace(prob, l=prob.l if prob.l.ndim == 1 else prob.l[:, 0].copy(),
                                  u=prob.u if prob.u.ndim == 1 else prob.u[:, 0].copy())
        c = pk.from_problem(one, dtype=pk.SUPPY_HALF_AUTO)
        fmt[spec["name"]] = "f16" if c.suppy_info_get()["a_dtype"] == pk.SUPPY_F16 else "bf16"
        c.close()
    batched["formats"] = fmt
    batched32, per_b32 = _serve_batched(pk, mats, reqs, pk.SUPPY_F32)
    # one at a time, FP32, per-matrix context resident after first use
    ctxs = {}
    lat1, fin1, queue1, service1, per_1, hist_1 = [], [], [], [], [], []
    t1 = time.perf_counter()
    for k, (ta, mi, l, u) in enumerate(reqs):
        while time.perf_counter() - t1 < ta:
            time.sleep(1e-4)
        ts = time.perf_counter() - t1
        prob, spec = mats[mi]
        if mi not in ctxs:
            q = _with_bounds(prob, l, u)
            ctxs[mi] = pk.from_problem(q, obj=spec["obj"], mode=spec["mode"])
        ctx = ctxs[mi]
        ctx.suppy_set_bounds(np.ascontiguousarray(l, np.float32), np.ascontiguousarray(u, np.float32))
        ctx.suppy_set_x(np.zeros(prob.A.n, np.float32))
        st = ctx.suppy_run(pk.suppy_params_default(**spec["sup"], **SERVE_STOP))[0]
        d = time.perf_counter() - t1
        ph, fh = ctx.suppy_history()
        lat1.append(d - ta)
        queue1.append(ts - ta)
        service1.append(d - ts)
        fin1.append(d)
        per_1.append((st["proximity"], st["objective"], st["sweeps"]))
        hist_1.append((ph.copy(), fh.copy()))
    for c in ctxs.values():
        c.close()
    torch.cuda.synchronize()
    plain = {"solves_per_s": len(reqs) / max(fin1), "p50_s": float(np.percentile(lat1, 50)),
             "p99_s": float(np.percentile(lat1, 99)), "makespan_s": max(fin1),
             "queue_p50_s": float(np.percentile(queue1, 50)),
             "queue_p99_s": float(np.percentile(queue1, 99)),
             "service_p50_s": float(np.percentile(service1, 50)),
             "service_p99_s": float(np.percentile(service1, 99)), "dtype": "f32"}

    def diffs(per_b):
        rp, ro, rp_eq, other_stop = [], [], [], 0
        for (pb, ob, sb), (p1, o1, s1), (h1, f1) in zip(per_b, per_1, hist_1):
            rp.append(abs(pb - p1) / max(abs(p1), 1e-300))
            ro.append(abs(ob - o1) / max(abs(o1), 1e-300))
            if sb != s1:
                other_stop += 1
            k = min(sb, len(h1)) - 1
            rp_eq.append(abs(pb - h1[k]) / max(abs(h1[k]), 1e-300) if k >= 0 else 0.0)
        miss = [i for i, (a, b) in enumerate(zip(rp, ro)) if a > 1e-3 or b > 1e-3]
        return {"final_proximity_rel_diff": {"median": float(np.median(rp)), "max": float(np.max(rp))},
                "final_objective_rel_diff": {"median": float(np.median(ro)), "max": float(np.max(ro))},
                "proximity_rel_diff_at_equal_sweeps": {"median": float(np.median(rp_eq)),
                                                       "max": float(np.max(rp_eq))},
                "requests_stopping_at_another_sweep": other_stop,
                "requests_above_1e-3": len(miss),
                "requests_above_1e-3_stopping_elsewhere": sum(1 for i in miss if per_b[i][2] != per_1[i][2]),
                "requests_above_1e-3_by_matrix": by_matrix(miss),
                "proximity_above_1e-3": sum(1 for a in rp if a > 1e-3)}

    def by_matrix(idx):
        out = {}
        for i in idx:
            nm = mats[reqs[i][1]][1]["name"]
            out[nm] = out.get(nm, 0) + 1
        return out

    batched.update(diffs(per_b))
    batched32.update(diffs(per_b32))
    return {"requests": len(reqs), "arrival_rate_per_s": 200.0,
            "arrivals_span_s": reqs[-1][0],
            "mix": {spec["name"]: sum(1 for r in reqs if r[1] == i)
                    for i, (_, spec) in enumerate(mats)},
            "batched": batched, "batched_f32": batched32, "one_at_a_time": plain,
            "stopping": "proximity change < 1e-4 relative for 5 sweeps, P <= 1e-6, or 500 sweeps"}


def _with_bounds(prob, l, u):
    import copy
    q = copy.copy(prob)
    q.l, q.u = np.ascontiguousarray(l, np.float32), np.ascontiguousarray(u, np.float32)
    return q


def ours(args):
    import torch
    rank, world, local = dist_env()
    K, W = args.steps, args.warmup
    prob = ct512()
    A = prob.A
    cpu = None
    if rank == 0 and not args.no_cpu:
        # before the first CUDA call: the all-cores oracle arm forks its workers
        cpu = cpu_baselines(prob, args.cpu_seconds)
        _ORACLE.clear()
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("gloo")
    torch.cuda.set_device(local)
    from paper_2606_27086_gb300 import build as pkbuild
    pkbuild.build()
    import paper_2606_27086_gb300 as pk

    log(f"[bench] CT 512^2: m={A.m} n={A.n} nnz={A.nnz}")
    # the sweep strategy and its launch shapes are chosen by the library's
    # tuner at create (outside the timed region): one pass with L2
    # reductions, two passes over CSR and CSC copies, or the tiled one pass
    t0 = time.perf_counter()
    if args.pin:
        # a configuration the tuner chose in a plain run, rebuilt without
        # timing (under a profiler the tuner's timings are not the plain ones)
        ctx = pk.from_problem(prob, obj=pk.SUPPY_OBJ_TV_ISO, **pinned_opts(pk, args.pin))
    else:
        ctx = pk.from_problem(prob, obj=pk.SUPPY_OBJ_TV_ISO, tune=1)
    t_create = time.perf_counter() - t0
    x_reset = torch.zeros(A.n, dtype=torch.float32, device="cuda")
    p_solve = pk.suppy_params_default(max_sweeps=SWEEPS, **SUP)

    def solve():
        ctx.suppy_set_x(x_reset)                 # box(0): a new solve
        ctx.suppy_run(p_solve, want_stats=False)  # 200 iterations, enqueued

    for _ in range(W):
        solve()
    torch.cuda.synchronize()
    if world > 1:
        torch.distributed.barrier()
    sampler = ClockSampler(gpu_id_for(local))
    sampler.start()
    time.sleep(0.3)
    nvtx = getattr(torch.cuda, "nvtx", None)
    if nvtx:
        nvtx.range_push("timed")
    l0 = ctx.suppy_launch_count()
    s = torch.cuda.current_stream()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record(s)
    for _ in range(K):
        solve()
    e1.record(s)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    nl = ctx.suppy_launch_count() - l0
    if nvtx:
        nvtx.range_pop()
    clocks = sampler.stop()
    st = ctx.suppy_run(pk.suppy_params_default(max_sweeps=0, **SUP))
    # per-kernel times: one more solve with CUDA events around every launch
    ctx.suppy_set_x(x_reset)
    _, kt, _ = time_iterations(ctx, pk, SWEEPS, 0, SUP, with_timing=True)
    ms, value = aggregate_over_ranks(ms, A.nnz * SWEEPS * K, world)
    info, per, t_sweep = summarize(ctx, prob, SWEEPS, kt, 4)
    peak, peak_kind = peaks()
    alg = sweep_alg_bytes(A.m, A.n, A.nnz, 4)
    achieved = alg / (t_sweep * 1e-3) / 1e9
    traffic, tnote = sweep_traffic(info)
    roof = {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
            "frac": achieved / peak, "traffic": traffic,
            "kernel": "sweep (every launch of one application of T: " + STRATEGY[info["strategy"]] +
                      (", patch numbering" if info.get("scatter_patch") else "") + ")",
            "alg_bytes_per_launch": alg, "launch_ms": t_sweep,
            "alg_bytes_formula": "nnz*(4+4) + m*16 + n*16 per sweep",
            "peak_source": peak_kind + " (MEASURED_PEAKS hbm_gbs, a burst copy)"}
    if tnote:
        roof["traffic_note"] = tnote

    # end to end through the C ABI with host buffers: per step new slab bounds
    # and x0 from pinned host memory, one solve, x back to pinned host memory
    Ke = max(3, min(K, 10))
    l_pin = torch.from_numpy(np.ascontiguousarray(prob.l)).pin_memory()
    u_pin = torch.from_numpy(np.ascontiguousarray(prob.u)).pin_memory()
    x0_pin = torch.zeros(A.n, dtype=torch.float32).pin_memory()
    x_pin = torch.empty(A.n, dtype=torch.float32).pin_memory()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(Ke):
        ctx.suppy_update_bounds_async(l_pin, u_pin)
        ctx.suppy_set_x(x0_pin)
        ctx.suppy_run(p_solve, want_stats=False)
        ctx.suppy_get_x(x_pin)
    torch.cuda.synchronize()
    te = time.perf_counter() - t0
    e2e = {"value": A.nnz * SWEEPS * Ke * world / te, "unit": UNIT,
           "h2d_bytes_per_step": 2 * A.m * 4 + A.n * 4, "d2h_bytes_per_step": A.n * 4 + 40,
           "steps": Ke,
           "note": "per step (one solve): suppy_update_bounds_async (pinned host l, u), "
                   "suppy_set_x (pinned host x0; the solve starts at box(0)), suppy_run of "
                   f"{SWEEPS} superiorized iterations (enqueued), suppy_get_x (pinned host x: "
                   "the step's one synchronization)"}

    res = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": K,
           "warmup": W, "ms_per_step": ms / K, "higher_is_better": True, "scaling": "weak",
           "vs_baseline": None, "dtype": "f32", "data": "synthetic", "config": config_of(prob),
           "roofline": roof, "kernels": per, "e2e": e2e,
           "gpu_launches": int(nl), "clocks": clocks, "create_s": t_create,
           "sweeps_per_step": SWEEPS,
           "launch_shape": {k: info[k] for k in ("strategy", "block", "scatter", "tma", "tiles", "chunks",
                                                  "tile_warps1", "tile_warps2", "tile_coef_warps",
                                                  "tile_ring", "tile_stream_bytes",
                                                  "tile_segments", "tile", "stages", "col_tile",
                                                  "col_stages", "map", "col_map",
                                                  "lanes_per_row", "col_lanes",
                                                  "transposed_rows", "scatter_patch",
                                                  "perturb_cluster")}}
    res["launch_shape"]["pin"] = pin_of(info)   # rebuilds it without timing
    if info["block"] == STRIP_BLOCK:
        # the shape of the streamed passes, which the strips do not run
        for k in ("tile", "stages", "col_tile", "col_stages", "map", "col_map"):
            res["launch_shape"].pop(k)
    if args.pin:
        res["launch_shape"]["pinned"] = args.pin
    ctx.close()
    if rank == 0 and not args.no_variants:
        res["variants"] = variants(pk, K, min(W, 5))
        res["precision"] = precision(pk)
    if rank == 0 and args.serve_requests > 0:
        res["serving"] = serving(pk, args.serve_requests)
    if cpu is not None:
        res["cpu_baseline"] = cpu
    if world > 1:
        torch.distributed.barrier()
    if rank == 0:
        detail = json.dumps(res)
        if args.detail:
            with open(args.detail, "w") as f:
                f.write(detail + "\n")
        else:
            log(f"[bench] detail {detail}")
        print(json.dumps(headline(res)), flush=True)
    return 0


def headline(res: dict) -> dict:
    """The result line: the whole record but for the secondary workloads, of which
    it keeps one figure each, so that it stays a line of about four kilobytes (the
    record itself, some 27, goes to stderr or --detail FILE)."""
    out = {k: v for k, v in res.items() if k not in ("variants", "precision", "serving", "cpu_baseline")}
    out["launch_shape"] = {k: v for k, v in res["launch_shape"].items() if v}
    if "variants" in res:
        out["variants"] = {k: float(f"{v['value']:.4g}") for k, v in res["variants"].items()
                           if isinstance(v, dict) and "value" in v}
    if "serving" in res:
        out["serving"] = {k: {q: float(f"{v[q]:.4g}") for q in ("solves_per_s", "p50_s", "p99_s") if q in v}
                          for k, v in res["serving"].items() if isinstance(v, dict) and "solves_per_s" in v}
    if "cpu_baseline" in res:
        out["cpu_baseline"] = {k: res["cpu_baseline"].get(k) for k in ("value", "unit", "cores", "kind")}
    return out


STRIP_BLOCK = 800   # threads per CTA of the strip-ordered passes (suppy_info.block)


def pin_of(info: dict) -> str:
    """The --pin of a context's launch configuration.  Strips have no shape to
    give: the strategy with every streaming option left open takes them."""
    if info["block"] == STRIP_BLOCK:
        return f"{info['strategy']},0,0,0,0,0,0"
    tr = 0 if info["strategy"] == 3 else (2 if info["scatter_patch"] else 1) if info["transposed_rows"] else -1
    return ",".join(str(v) for v in (info["strategy"], info["tile"], info["stages"],
                                     info["lanes_per_row"] if info["tma"] else 0, info["map"], info["col_map"], tr))


def pinned_opts(pk, pin: str) -> dict:
    """from_problem options of a --pin launch configuration
    (strategy,tile,stages,lanes,map,col_map[,pixel numbering]; zeros leave an
    option open)."""
    vals = [int(v) for v in pin.split(",")]
    st_, tile, stages, lanes, mp, cmp_ = vals[:6]
    tr = vals[6] if len(vals) > 6 else -1
    return dict(strategy=st_, stream_shape=(tile, stages, lanes), stream_map=mp,
                stream_col_map=cmp_, scatter_transpose=tr)


def profile_case(case: int, steps: int, warm: int = 0, pin: str = "") -> int:
    """A short run for ncu.  Cases 1 / 2: CT 384x384 (A ~0.4 GB, above L2; the
    device holds about 1 GB) with the one- / two-pass sweep.  Case 3: the CT
    512x512 workload with the sweep and launch shapes bench.py uses (two
    passes, shapes tuned at create); case 4: the same with the one-pass sweep;
    case 5: the horseshoe radiotherapy plan as a split problem (dose-volume
    sets by the CQ step, slabs by EMR, mean-dose perturbations); case 6: the
    CT 512x512 workload block-iteratively (36 interleaved angle blocks, tuned);
    case 7: the seismic workload with 16 right-hand sides (batched register-fed
    two-pass sweep, one perturbation cluster per image); case 8: CT 384x384
    with EMR and the variance rule evaluated every iteration (extrapolation
    and variance kernels); case 9: CT 384x384 with the register-fed two-pass
    sweep (no bulk copies), the cluster perturbation with the image in shared
    memory, and the standalone proximity and objective evaluations
    (two each, after the iterations); case 10: a 2048x2048 image over a
    random slab system (20000 rows) with TV, whose image exceeds a cluster's
    shared memory, so the cluster perturbation reads them from
    global memory; case 11: CT 384x384 with the tiled one-pass sweep.
    The profiled iterations run inside the NVTX range "profile", so that
    `ncu --nvtx --nvtx-include profile/` skips the tuning launches and the
    `warm` iterations run before it.  Cases 3, 4 and 6 take a --pin launch
    configuration instead of tuning (under ncu the serialised launches
    distort the tuner's timings)."""
    import torch
    import synth
    from paper_2606_27086_gb300 import build as pkbuild
    pkbuild.build()
    import paper_2606_27086_gb300 as pk
    params = SUP
    if case == 5:
        prob = synth.rt_split_problem()
        ctx = pk.from_problem(prob, obj=pk.SUPPY_OBJ_LINEAR, mode=pk.SUPPY_EMR)
        sp = prob.meta["split"]
        Aq = sp["Aq"]
        ctx.suppy_set_dvc(Aq.row_ptr, Aq.col, Aq.val, Aq.m, sp["sptr"], sp["dvcs"], 1.0)
        params = dict(gamma=1.0, alpha=0.7, n_red=1, restart_every=500)
    elif case == 6:
        prob = ct512()
        prob.blocks = synth.angle_blocks(360, 725, 36)
        kw = pinned_opts(pk, pin) if pin else dict(tune=1)
        ctx = pk.from_problem(prob, obj=pk.SUPPY_OBJ_TV_ISO, mode=pk.SUPPY_BIP, **kw)
    elif case == 7:
        prob = synth.seismic_problem(nrhs=16)
        ctx = pk.from_problem(prob, obj=pk.SUPPY_OBJ_TV_ANISO, strategy=pk.STRATEGY_TWO_PASS)
    elif case == 8:
        prob = synth.ct_problem(384, 270, 545, I0=5e3, delta=0.02, seed_phantom=201,
                                seed_noise=202)
        ctx = pk.from_problem(prob, obj=pk.SUPPY_OBJ_TV_ISO, mode=pk.SUPPY_EMR)
        params = dict(SUP, variance_tol=1e-30)
    elif case == 9:
        prob = synth.ct_problem(384, 270, 545, I0=5e3, delta=0.02, seed_phantom=201,
                                seed_noise=202)
        ctx = pk.from_problem(prob, obj=pk.SUPPY_OBJ_TV_ISO, strategy=pk.STRATEGY_TWO_PASS, tma=-1,
                              perturb_path=1)
    elif case == 10:
        prob = synth.random_problem(20000, 2048 * 2048, seed=11, feasible=False, mean_len=200)
        prob.shape = (2048, 2048)
        ctx = pk.from_problem(prob, obj=pk.SUPPY_OBJ_TV_ISO, strategy=pk.STRATEGY_TWO_PASS,
                              perturb_path=1)
    elif case == 11:
        prob = synth.ct_problem(384, 270, 545, I0=5e3, delta=0.02, seed_phantom=201,
                                seed_noise=202)
        ctx = pk.from_problem(prob, obj=pk.SUPPY_OBJ_TV_ISO, strategy=pk.STRATEGY_TILED)
    elif case in (3, 4):
        prob = ct512()
        kw = pinned_opts(pk, pin) if pin else dict(
            tune=1, strategy=pk.STRATEGY_TWO_PASS if case == 3 else pk.STRATEGY_ONE_PASS)
        ctx = pk.from_problem(prob, obj=pk.SUPPY_OBJ_TV_ISO, **kw)
    else:
        prob = synth.ct_problem(384, 270, 545, I0=5e3, delta=0.02, seed_phantom=201,
                                seed_noise=202)
        ctx = pk.from_problem(prob, obj=pk.SUPPY_OBJ_TV_ISO, strategy=case)
    if warm:
        # steady state first: the early phases spend many trials
        ctx.suppy_run(pk.suppy_params_default(max_sweeps=warm, **params))
    torch.cuda.synchronize()
    nvtx = getattr(torch.cuda, "nvtx", None)
    if nvtx:
        nvtx.range_push("profile")
    st = ctx.suppy_run(pk.suppy_params_default(max_sweeps=steps, use_graphs=0, **params))
    if case == 9:
        for _ in range(2):
            ctx.suppy_proximity()
            ctx.suppy_objective()
    torch.cuda.synchronize()
    if nvtx:
        nvtx.range_pop()
    info = ctx.suppy_info_get()
    log(f"[profile] case {case}: m={prob.A.m} n={prob.A.n} nnz={prob.A.nnz} "
        f"shape={info} state={st[0]} launches={ctx.suppy_launch_count()}")
    ctx.close()
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10,
                    help="timed solves (each 200 superiorized iterations from box(0))")
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--profile-warmup", type=int, default=0,
                    help="with --profile: unprofiled iterations before the profiled ones (300 "
                         "reaches the steady state; 0 profiles the first iterations)")
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-variants", action="store_true")
    ap.add_argument("--pin", default="",
                    help="build the headline context with this launch configuration instead of "
                         "tuning it: strategy,tile,stages,lanes,map,col_map[,pixel numbering: "
                         "1 column-major rows, 2 patches (one pass), -1 off] as a plain run's "
                         "launch_shape reports it under pin (e.g. 1,4096,6,32,2,2,2; "
                         "1,0,0,0,0,0,0 for strips), for runs under a profiler, whose serialised "
                         "launches distort the tuner's timings")
    ap.add_argument("--detail", default="", metavar="FILE",
                    help="write the whole record (secondary workloads, precision, serving) to FILE "
                         "instead of stderr; the result line on stdout is its short form")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--cpu-seconds", type=float, default=12.0)
    ap.add_argument("--serve-requests", type=int, default=512,
                    help="also run the serving mix with this many requests (512: the full "
                         "trace; 0 skips it) and report it under 'serving'")
    ap.add_argument("--profile", type=int, default=0, choices=list(range(12)),
                    help="run a short profiling case and exit: CT 384x384 (270 angles x 545 "
                         "bins) with sweep strategy 1 (one pass) or 2 (two passes), or the "
                         "CT 512x512 workload with tuned launch shapes: 3 two passes, 4 one "
                         "pass; 5 the horseshoe split problem (DVCs by the CQ step); 6 CT "
                         "512x512 with 36 BIP blocks; 7 seismic with 16 right-hand sides; 8 "
                         "CT 384x384 with EMR and the variance rule; 9 CT 384x384, "
                         "register-fed sweep, cluster perturbation, standalone proximity and "
                         "objective; 10 a 2048x2048 TV image, cluster perturbation from "
                         "global memory; 11 CT 384x384 with the tiled sweep")
    args = ap.parse_args()
    if args.profile:
        return profile_case(args.profile, args.steps if args.steps < 50 else 6,
                            args.profile_warmup, args.pin)
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        # each oracle step is about two seconds of CPU work: bound the sample
        args.steps = min(args.steps, 20)
        args.warmup = min(args.warmup, 3)
        return reference_arm(args)
    return ours(args)


if __name__ == "__main__":
    sys.exit(main())
