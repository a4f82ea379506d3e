#!/usr/bin/env python3
"""Benchmark of the TPMC hot path on GB300.

Workload (one step): the plate / closed-cylinder sweep -- a 1 x 1 m plate
(2 triangles) and a closed cylinder R = 0.5 m, L = 2 m (4,096 triangles), each
over 32 angles of attack in [0, 90] deg x S in {2, 5, 10} x {specular, diffuse}
re-emission, 1e7 particles per case (384 cases, 3.84e9 particles), atomic
oxygen at T_inf = 1000 K, T_W = 300 K, FP32 traversal with FP64 set-up and
reduction.  One step is four batched sweep calls (mesh x re-emission) of 96 cases
each: a set-up, batches of 2^26 particles seeded and traced by a persistent launch
each, and a reduction.

value: traced particles per second with meshes resident on the device (CUDA
events around each step on the launching stream; a 256 MiB L2 flush between
steps, outside the timed intervals).  e2e: the same metric through the public
API with host buffers (mesh upload and BVH build, host inputs, host results).
"""
from __future__ import annotations

import argparse
import hashlib
import json
import math
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

from tpmc_inputs import meshes as M  # noqa: E402
from tpmc_inputs import workloads as W  # noqa: E402

METRIC = "traced particles/s on 1 GB300 (% roofline); C_D err vs oracle; serve p50/p99 ms"
UNIT = "particles/s"
WORKLOAD = "plate(2 tri)+cylinder(4096 tri) sweep: 32 alpha x S{2,5,10} x {specular,diffuse}, 1e7 particles/case"
N_EACH = 10_000_000
FP32_LANES_PER_SM = 128
# Algorithmic work per unit of BVH ray casting (FMA = 2 flops; add, mul, min,
# max, compare = 1).  A node visit tests each of its child boxes (the node's
# width: 2 for the binary tree, up to 8 for the compressed wide tree) and reads
# the node once (64 B binary, 80 B compressed wide); the counts of node visits
# and triangle tests are measured per run.
FLOPS_PER_CHILD_BOX = 20     # slab test of one child box: 6 FMA + 8 min/max/compare
FLOPS_PER_TRI_TEST = 35      # watertight test: translate, shear, 3 edge functions, det, T
FLOPS_PER_PARTICLE = 150     # seeding: two inverse-CDF solves, Box-Muller, two rotations
FLOPS_PER_HIT = 30           # re-emission, momentum difference, torque, quantisation
BYTES_PER_TRI_TEST = 48      # three float4 vertices
# DRAM bytes per sweep call from an ncu capture, valid only for the kernel source,
# its build flags, the BVH builder and the host code that decides on the pool, its
# batches and its entries it was taken with (keyed by the SHA-256 of TRAFFIC_SOURCES
# in that order).
TRAFFIC_SOURCES = ("csrc/trace.cuh", "csrc/trace_w2.cu", "csrc/kernels.cu", "csrc/bvh.cpp", "build.py", "csrc/api.cpp",
                   "csrc/runtime.h", "csrc/tpmc_internal.h")
# Mean over the four bench groups of dram__bytes_read.sum + dram__bytes_write.sum
# over the seeding and trace launches of one full-size call (9.6e8 particles).
TRACE_TRAFFIC = {"98a95d7d657a0f1f2ce67b82a03d21c50748c6b69311e25a83394fe2fed13a5d": 25_431_364_480}


def kernel_source_hash() -> str:
    h = hashlib.sha256()
    for name in TRAFFIC_SOURCES:
        with open(os.path.join(ROOT, "paper_1312_3691_gb300", name), "rb") as f:
            h.update(f.read())
    return h.hexdigest()


def launches_per_call(particles: int) -> int:
    """Kernels of one sweep call of this size: the set-up, a seeding and a trace launch for every batch of the pool
    (2^26 particles, the full size, which a device with nothing else on it has room for), and the reduction."""
    return 2 + 2 * -(-particles // (1 << 26))


def rank_stream_base(rank: int, group: int) -> int:
    """Philox stream id of a sweep group on a rank: ranks trace independent
    particle streams of the same workload (weak scaling, no data exchange)."""
    return rank * 4096 + group * 128


def max_over_ranks(value: float, dist, device) -> float:
    """The slowest rank's time (the job's time) when several ranks run."""
    if dist is None:
        return value
    import torch

    t = torch.tensor([value], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def groups():
    """The four sweep groups of one step: (shape, eps, xyz, tri, base params, dirs[96], S[96])."""
    out = []
    for shape in ("plate", "cylinder"):
        for eps in (0.0, 1.0):
            xyz, tri, cases = W.sweep_cases(shape, N_each=N_EACH, eps_values=(eps,))
            dirs = np.array([c["params"]["dir"] for c in cases])
            S = np.array([c["S"] for c in cases])
            base = dict(cases[0]["params"])
            out.append(dict(shape=shape, eps=eps, xyz=xyz, tri=tri, base=base, dirs=dirs, S=S, cases=cases))
    return out


class ClockSampler:
    """nvidia-smi sampling of SM clocks and throttle reasons during the timed region."""

    FIELDS = "index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown," \
             "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown," \
             "clocks_event_reasons.sw_power_cap"

    def __init__(self, device_index: int):
        self.dev = device_index
        self.proc = None
        self.lines = []
        self.thread = None

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.dev}", f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
            return
        self.thread = threading.Thread(target=self._read, daemon=True)
        self.thread.start()

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        if self.thread:
            self.thread.join(timeout=5)
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for n, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(n)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def roofline_of(parts, seconds: float, ceil: dict) -> dict:
    """The trace kernel's roofline for one measured run: particles/s against
    min(B_L2 / bytes per particle, P_FP32 / flops per particle), with B_L2 and
    P_FP32 the ceilings measured on this device (tpmc_measure_ceilings).  The
    kernel reads nodes and triangles that stay in L1/L2, so L2 bandwidth, not
    HBM, is the memory ceiling.  `parts` lists (work, node bytes, BVH width) of
    the launches timed together in `seconds`; `achieved` is in the binding
    ceiling's unit."""
    tot = {"particles": 0, "hits": 0, "nodes": 0, "tris": 0}
    flops = l2_bytes = 0.0
    widths = set()
    for work, node_bytes, width in parts:
        for k in tot:
            tot[k] += work[k]
        flops += (FLOPS_PER_CHILD_BOX * width * work["nodes"] + FLOPS_PER_TRI_TEST * work["tris"] +
                  FLOPS_PER_PARTICLE * work["particles"] + FLOPS_PER_HIT * work["hits"])
        l2_bytes += node_bytes * work["nodes"] + BYTES_PER_TRI_TEST * work["tris"]
        widths.add((width, node_bytes))
    n = max(tot["particles"], 1)
    fpp, bpp = flops / n, l2_bytes / n
    rate = tot["particles"] / seconds
    bound_l2 = ceil["l2_read_gbs"] * 1e9 / max(bpp, 1e-30)
    bound_fp32 = ceil["fp32_tflops"] * 1e12 / max(fpp, 1e-30)
    if bound_l2 <= bound_fp32:
        out = {"bound": "l2", "achieved": rate * bpp / 1e9, "peak": ceil["l2_read_gbs"], "unit": "GB/s"}
    else:
        out = {"bound": "fp32", "achieved": rate * fpp / 1e12, "peak": ceil["fp32_tflops"], "unit": "TFLOP/s"}
    out["frac"] = rate / min(bound_l2, bound_fp32)
    out.update({
        "particles_per_s": rate, "flops_per_particle": fpp, "bytes_per_particle": bpp, "work": tot,
        "node_visits_per_particle": tot["nodes"] / n, "tri_tests_per_particle": tot["tris"] / n,
        "hits_per_particle": tot["hits"] / n,
        "bvh": [{"width": w, "node_bytes": b} for w, b in sorted(widths)],
        "particles_per_s_l2_bound": bound_l2, "particles_per_s_fp32_bound": bound_fp32,
        "fp32_frac": rate * fpp / (ceil["fp32_tflops"] * 1e12), "l2_frac": rate * bpp / (ceil["l2_read_gbs"] * 1e9),
        "ceilings": {"l2_read_gbs": ceil["l2_read_gbs"], "fp32_tflops": ceil["fp32_tflops"],
                     "basis": "measured on this device: L2-resident streaming read (32 MiB, 64 passes, L1 "
                              "bypassed) and an FP32 FMA loop, best of 5 (tpmc_measure_ceilings)"},
        "units": {"flops_per_child_box": FLOPS_PER_CHILD_BOX, "flops_per_tri_test": FLOPS_PER_TRI_TEST,
                  "flops_per_particle": FLOPS_PER_PARTICLE, "flops_per_hit": FLOPS_PER_HIT,
                  "bytes_per_tri_test": BYTES_PER_TRI_TEST},
    })
    return out


def work_of(results) -> dict:
    w = {"particles": 0, "hits": 0, "nodes": 0, "tris": 0}
    for r in results:
        w["particles"] += r["n_particles"]
        w["hits"] += r["n_hits"]
        w["nodes"] += r["n_node_visits"]
        w["tris"] += r["n_tri_tests"]
    return w


def measured_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f)
    except OSError:
        return {}


# ---------------------------------------------------------------- CPU side
def cpu_baseline_leg(T, ctx, results_by_group):
    """The bench's CPU-baseline leg, the one place besides `--impl reference`
    where it runs the oracle: after the timed region, on rank 0, it times the
    oracle on the host cores and, on the same oracle runs, states the GPU
    results' C_D error (all sweep cases; C1 and C3 on shared particles) and the
    per-particle path parity of C1-C4."""
    cpu_base, cd_err = cpu_baseline_and_cd_error(results_by_group)
    return cpu_base, cd_err, other_configs_vs_oracle(T, ctx), parity_excused_shares(T, ctx)


def cpu_baseline_and_cd_error(results_by_group, budget_s=12.0):
    """The FP64 oracle timed on the host cores on a bounded sample of the same
    workload, and the C_D error of the GPU results against the oracle's exact
    (panel-sum) expectation for every case."""
    import oracle

    oracle.build()
    threads = os.cpu_count() or 1
    gs = groups()
    rates = {}
    sample_desc = []
    for shape, per_case in (("plate", 250_000), ("cylinder", 60_000)):
        t_total, n_total = 0.0, 0
        for g in gs:
            if g["shape"] != shape:
                continue
            om = oracle.Mesh(g["xyz"], g["tri"])
            for ci in (10, 50):
                c = g["cases"][ci]
                p = oracle.make_params(**c["params"], threads=threads)
                t0 = time.perf_counter()
                oracle.trace(om, p, c["N"], pid_begin=0, count=per_case)
                t_total += time.perf_counter() - t0
                n_total += per_case
        rates[shape] = n_total / t_total
        sample_desc.append(f"{shape}: first {per_case} ids of 4 cases")
    # the oracle's own median-split BVH on the cylinder (intersect=2), beside its
    # default there (brute force over all triangles for meshes of <= 5,000)
    t_bvh, n_bvh = 0.0, 0
    for g in gs:
        if g["shape"] != "cylinder":
            continue
        om = oracle.Mesh(g["xyz"], g["tri"])
        for ci in (10, 50):
            c = g["cases"][ci]
            p = oracle.make_params(**c["params"], threads=threads, intersect=2)
            t0 = time.perf_counter()
            oracle.trace(om, p, c["N"], pid_begin=0, count=4 * 60_000)
            t_bvh += time.perf_counter() - t0
            n_bvh += 4 * 60_000
    rate_cyl_bvh = n_bvh / t_bvh
    # the workload traces equal particle counts on both meshes
    rate = 1.0 / (0.5 / rates["plate"] + 0.5 / rates["cylinder"])
    rate_bvh = 1.0 / (0.5 / rates["plate"] + 0.5 / rate_cyl_bvh)
    cd = None
    if results_by_group is not None:
        zs, rels, within = [], [], []
        for g, res in zip(gs, results_by_group):
            for c, r in zip(g["cases"], res):
                Vhat = np.asarray(c["params"]["dir"])
                F = oracle.panel_sum(g["xyz"], g["tri"], Vhat, c["S"], c["eps"], math.sqrt(300.0 / 1000.0),
                                     two_sided=(g["shape"] == "plate"))
                ref = F @ Vhat / (0.5 * c["S"] ** 2 * c["params"]["A_ref"])
                err = abs(r["CD"] - ref)
                if r["CD_sigma"] > 0:
                    zs.append(err / r["CD_sigma"])
                # 1e-12: the flow edge-on to the specular plate, where drag and sigma both vanish
                within.append(err <= 1e-4 * abs(ref) + 3.0 * r["CD_sigma"] + 1e-12)
                rels.append(err / max(abs(ref), 1e-12))
        cd = {"reference": "oracle panel-sum expectation (exact for these convex meshes)",
              "n_cases": len(rels), "max_abs_z": max(zs) if zs else None,
              "frac_within_3sigma_plus_1e-4": float(np.mean(within)),
              "max_rel": max(rels), "median_rel": float(np.median(rels))}
    base = {"value": rate, "unit": UNIT, "cores": threads, "kind": "oracle",
            "sample": "; ".join(sample_desc) + f"; plate {rates['plate']:.4g}/s, cylinder {rates['cylinder']:.4g}/s,"
                      " combined for equal particle counts",
            "intersection": {"plate": "brute force over its 2 triangles (the oracle's default below 5,000)",
                             "cylinder": "brute force over its 4,096 triangles (the oracle's default below 5,000)"},
            "cylinder_oracle_bvh_particles_per_s": rate_cyl_bvh,
            "value_with_oracle_bvh_on_cylinder": rate_bvh,
            "bvh_sample": "cylinder: first 240,000 ids of 4 cases with the oracle's median-split BVH (intersect=2)"}
    return base, cd


def other_configs_vs_oracle(T, ctx):
    """C_D of the sphere (FP64, 1e5 particles) and of the concave satellite (FP32,
    the first 1e5 particle ids) against the oracle on the same particles, with the
    oracle's rate on them (host cores)."""
    import oracle

    oracle.build()
    threads = os.cpu_count() or 1
    out = {}
    c1 = W.icosphere_case(N=100_000)
    c3 = W.satellite_case(N=100_000)
    for name, case, prec in (("C1_icosphere_fp64_1e5", c1, T.TPMC_FP64), ("C3_satellite_fp32_1e5", c3, T.TPMC_FP32)):
        mesh = T.tpmc_mesh_load(ctx, case["xyz"], case["tri"])
        try:
            g = T.tpmc_trace(ctx, mesh, T.make_params(**case["params"], precision=prec), case["N"])
        finally:
            T.tpmc_mesh_unload(ctx, mesh)
        om = oracle.Mesh(case["xyz"], case["tri"])
        t0 = time.perf_counter()
        o, _, _ = oracle.trace(om, oracle.make_params(**case["params"], threads=threads), case["N"])
        t_orc = time.perf_counter() - t0
        row = {"gpu_CD": g["CD"], "oracle_CD": o["CD"], "CD_sigma": o["CD_sigma"],
               "rel_diff": abs(g["CD"] - o["CD"]) / abs(o["CD"]),
               "torque_rel_diff": float(np.linalg.norm(np.asarray(g["torque"]) - o["torque"]) /
                                        max(np.linalg.norm(o["torque"]), 1e-300)),
               "gpu_ms": g["ms"], "oracle_particles_per_s": case["N"] / t_orc, "oracle_cores": threads}
        if name.startswith("C1"):
            Vhat = np.asarray(case["params"]["dir"])
            F = oracle.panel_sum(case["xyz"], case["tri"], Vhat, 7.5, 1.0, math.sqrt(0.3))
            row["exact_faceted_CD"] = float(F @ Vhat / (0.5 * 7.5 ** 2 * math.pi))
        out[name] = row
    return out


def parity_excused_shares(T, ctx):
    """Path parity on the same Philox streams for C1-C4 (after the timed region):
    the share of particles whose hit paths differ from the oracle's after a
    near-edge or grazing hit (excused), binned by the bounce where they first
    differ, the count that differ away from edges (must be 0), and the FP32
    momentum parity of the identical-path particles."""
    import oracle

    from tests.parity_util import dv_parity, path_stats

    oracle.build()
    threads = os.cpu_count() or 1
    K = 16
    c_mp = (2 * W.K_B * 1000.0 / W.M_OXYGEN) ** 0.5
    cases = []
    c1 = W.icosphere_case(N=100_000)
    cases.append(("C1_icosphere_fp64", c1["xyz"], c1["tri"], [(c1["params"], T.TPMC_FP64, 0, 100_000)]))
    for shape in ("plate", "cylinder"):
        xyz, tri, cs = W.sweep_cases(shape, N_each=N_EACH, n_alpha=32)
        runs = [(cs[i]["params"], T.TPMC_FP32, 0, 50_000) for i in (len(cs) - 20, 45)]
        cases.append((f"C2_{shape}_fp32", xyz, tri, runs))
    c3 = W.satellite_case(N=1)
    cases.append(("C3_satellite_fp32", c3["xyz"], c3["tri"], [(c3["params"], T.TPMC_FP32, 0, 100_000)]))
    grid = W.attitude_grid(32, 32)
    runs = []
    for k in (5, 300, 517, 1000):
        pk = dict(c3["params"], dir=tuple(grid[k]), V=7.5 * c_mp)
        runs.append((pk, T.TPMC_FP32, (1 << 20) + 1024 + k, 25_000))
    cases.append(("C4_attitude_items_fp32", c3["xyz"], c3["tri"], runs))
    out = {}
    for name, xyz, tri, runs in cases:
        mesh = T.tpmc_mesh_load(ctx, xyz, tri)
        om = oracle.Mesh(xyz, tri)
        agg = {"n": 0, "identical": 0, "excused": 0, "unexplained": 0, "excused_by_bounce": [0] * K}
        dvs = []
        try:
            for params, prec, stream, n in runs:
                _, rec = T.tpmc_trace_records(ctx, mesh, T.make_params(**params, precision=prec, stream_id=stream),
                                              n, K=K)
                _, _, orec = oracle.trace(om, oracle.make_params(**params, stream=stream, threads=threads), n,
                                          records=True, K=K)
                st = path_stats(rec, orec, K)
                for k in ("n", "identical", "excused", "unexplained"):
                    agg[k] += st[k]
                agg["excused_by_bounce"] = [a + b for a, b in zip(agg["excused_by_bounce"], st["excused_by_bounce"])]
                dvs.append(dv_parity(rec, orec, st["_identical_mask"], params["dir"]))
        finally:
            T.tpmc_mesh_unload(ctx, mesh)
        agg["excused_share"] = agg["excused"] / max(agg["n"], 1)
        last = max([i for i, x in enumerate(agg["excused_by_bounce"]) if x] or [0])
        agg["excused_by_bounce"] = agg["excused_by_bounce"][:last + 1]
        agg["dv_identical_paths"] = {"median_rel_max": max(d.get("median_rel", 0.0) for d in dvs),
                                     "p99_rel_max": max(d.get("p99_rel", 0.0) for d in dvs),
                                     "drag_rel_max": max(d["drag_rel"] for d in dvs)}
        out[name] = agg
    return out


def run_reference(args):
    """Reference arm: the FP64 oracle timed as it stands on the host cores."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    import oracle

    oracle.build()
    threads = os.cpu_count() or 1
    gs = groups()
    meshes = {g["shape"]: oracle.Mesh(g["xyz"], g["tri"]) for g in gs}
    sample = {"plate": 60_000, "cylinder": 15_000}

    def step(k):
        t = {"plate": 0.0, "cylinder": 0.0}
        n = {"plate": 0, "cylinder": 0}
        for g in gs:
            c = g["cases"][(7 * k + 3) % len(g["cases"])]
            p = oracle.make_params(**c["params"], threads=threads)
            t0 = time.perf_counter()
            oracle.trace(meshes[g["shape"]], p, c["N"], pid_begin=0, count=sample[g["shape"]])
            t[g["shape"]] += time.perf_counter() - t0
            n[g["shape"]] += sample[g["shape"]]
        return t, n

    for k in range(args.warmup):
        step(k)
    tp = tc = 0.0
    np_ = nc = 0
    t_start = time.perf_counter()
    for k in range(args.steps):
        t, n = step(args.warmup + k)
        tp += t["plate"]; tc += t["cylinder"]; np_ += n["plate"]; nc += n["cylinder"]
    wall = time.perf_counter() - t_start
    rate = 1.0 / (0.5 / (np_ / tp) + 0.5 / (nc / tc))
    line = {
        "impl": "reference", "metric": METRIC, "value": rate, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * wall / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic", "config": {"workload": WORKLOAD, "particles_per_case": N_EACH},
        "cpu_baseline": {"value": rate, "unit": UNIT, "cores": threads, "kind": "oracle",
                         "sample": f"per step: first {sample['plate']} ids of 2 plate cases and "
                                   f"{sample['cylinder']} ids of 2 cylinder cases; rates combined for equal counts"},
        "e2e": {"value": rate, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


# ----------------------------------------------------- other configurations
def measure_satellite(T, ctx, torch, stream, ceil, target_triangles=60_000):
    """Concave synthetic satellite (60,656 or 503,537 triangles), 1e8 particles,
    <= 64 bounces, Maxwell 0.9 diffuse, per-panel pressure and shear: the host
    API's wall clock, and CUDA events on the library's stream around the same
    call for the roofline (work counted in a separate pass of the same query)."""
    case = W.satellite_case(N=100_000_000, target_triangles=target_triangles)
    mesh = T.tpmc_mesh_load(ctx, case["xyz"], case["tri"])
    info = T.tpmc_mesh_info(ctx, mesh)
    try:
        T.tpmc_set_stream(ctx, stream)
        p = T.make_params(**case["params"], want_panels=True)
        T.tpmc_trace(ctx, mesh, T.make_params(**case["params"]), 1_000_000)  # warm-up
        T.tpmc_set_counters(ctx, True)
        rc = T.tpmc_trace(ctx, mesh, T.make_params(**case["params"]), case["N"])
        T.tpmc_set_counters(ctx, False)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        r = T.tpmc_trace(ctx, mesh, p, case["N"])
        b.record(stream)
        torch.cuda.synchronize()
        gpu_ms = a.elapsed_time(b)
        pres, shear = T.tpmc_panels(ctx, r["query_id"], case["tri"].shape[0])
    finally:
        T.tpmc_mesh_unload(ctx, mesh)
    assert rc["sum_dv_q"] == r["sum_dv_q"]
    return {"workload": case["name"] + ", 1e8 particles, <=64 bounces, eps 0.9, panels",
            "particles_per_s": case["N"] / (r["ms"] / 1e3), "ms": r["ms"], "gpu_ms": gpu_ms,
            "CD": r["CD"], "CD_sigma": r["CD_sigma"],
            "torque_Nm": r["torque"], "hits_per_particle": r["n_hits"] / r["n_particles"],
            "truncated": r["n_truncated"], "max_abs_pressure_Pa": float(np.abs(pres).max()),
            "max_shear_Pa": float(shear.max()),
            "roofline": roofline_of([(work_of([rc]), info["node_bytes"], info["bvh_width"])], gpu_ms / 1e3, ceil)}


def measure_hemisphere(T, ctx):
    """Concave hemispherical shell (6,048 triangles) in a hyperthermal axial flow,
    1e8 particles, full diffuse accommodation: eps_eff = (C_D - 2) S_W / sqrt(pi)
    against Pratt's eps_D(90 deg) = 1.05349 (host API, wall clock)."""
    case = W.hemisphere_case(N=100_000_000)
    mesh = T.tpmc_mesh_load(ctx, case["xyz"], case["tri"])
    try:
        p = T.make_params(**case["params"])
        T.tpmc_trace(ctx, mesh, p, 1_000_000)  # warm-up
        r = T.tpmc_trace(ctx, mesh, p, case["N"])
    finally:
        T.tpmc_mesh_unload(ctx, mesh)
    k = case["S_W"] / math.sqrt(math.pi)
    return {"workload": case["name"] + ", 1e8 particles, diffuse",
            "particles_per_s": case["N"] / (r["ms"] / 1e3), "ms": r["ms"], "CD": r["CD"], "CD_sigma": r["CD_sigma"],
            "eps_eff": (r["CD"] - 2.0 - 1.0 / case["S"] ** 2) * k, "eps_eff_sigma": r["CD_sigma"] * k,
            "eps_D_pratt": 1.05349, "hits_per_hit_particle": r["n_hits"] / max(r["n_hit_particles"], 1)}


def measure_box_cv(T, ctx):
    """Sphere (1,280-triangle icosphere), S 5, diffuse, 1e7 particles per case, as the
    stream turns from a box face normal to a box diagonal: C_D of the flux-weighted
    box and of the Maxwell box relative to the spherical CV's C_D (the consistent
    seeding), with the combined standard error (host API, wall clock)."""
    xyz, tri = M.icosphere(3)
    N = 10_000_000
    mesh = T.tpmc_mesh_load(ctx, xyz, tri)
    rows, ms, n = [], 0.0, 0
    try:
        for alpha in (0.0, 15.0, 30.0, 45.0):
            a = math.radians(alpha)
            base = dict(**W.base_state(S=5.0), dir=(math.sin(a), 0.0, math.cos(a)), eps_diffuse=1.0, A_ref=math.pi,
                        seed=77, max_bounces=8)
            res = {}
            for name, extra in (("sphere", dict(r_cv=1.2)),
                                ("box_flux", dict(cv_kind=1, box_lo=(-1.2,) * 3, box_hi=(1.2,) * 3)),
                                ("box_maxwell", dict(cv_kind=2, box_lo=(-1.2,) * 3, box_hi=(1.2,) * 3))):
                res[name] = T.tpmc_trace(ctx, mesh, T.make_params(**base, **extra), N)
                ms += res[name]["ms"]
                n += N
            sph = res["sphere"]
            row = {"alpha_deg": alpha, "CD_sphere_cv": sph["CD"]}
            for name in ("box_flux", "box_maxwell"):
                r = res[name]
                row[name + "_vs_sphere_pct"] = 100.0 * (r["CD"] / sph["CD"] - 1.0)
                row[name + "_sigma_pct"] = 100.0 * math.hypot(r["CD_sigma"], sph["CD_sigma"]) / sph["CD"]
            rows.append(row)
    finally:
        T.tpmc_mesh_unload(ctx, mesh)
    return {"workload": "icosphere 1,280 tri, S 5, T_W/T_inf 0.3, diffuse, 1e7 particles per case; "
                        "CV: sphere r 1.2 m or box half-width 1.2 m",
            "particles_per_s": n / (ms / 1e3), "rows": rows}


def measure_moment_sweep(T, ctx, torch, stream, dev):
    """Restoring moment about the quarter chord (§III.D.1) on the synthetic
    satellite at the Table 1 conditions: alpha in [-90, 90] step 10 x 8 roll
    angles = 152 attitudes x 2^22 particles in one sweep call; the
    pitching-moment coefficient C_m = -M.e_p / (q_inf c) (pitch-up positive, area-
    scaled, A_ref = 1 m^2) for the horizontal (beta 0) and vertical (beta 90) rolls."""
    case = W.satellite_moment_case(N=1)
    alphas = [-90.0 + 10.0 * i for i in range(19)]
    betas = [45.0 * j for j in range(8)]
    V, E, grid = W.alpha_beta_dirs(alphas, betas)
    K, N_each = len(grid), 1 << 22
    mesh = T.tpmc_mesh_load(ctx, case["xyz"], case["tri"])
    try:
        base = T.make_params(**case["params"], stream_id=1 << 21)
        dd = torch.tensor(V, dtype=torch.float64, device=dev)
        out = torch.zeros(K * T.RESULT_BYTES, dtype=torch.uint8, device=dev)
        T.tpmc_set_stream(ctx, stream)
        T.tpmc_sweep_device(ctx, mesh, base, dd[:8], None, 8, 1 << 16, out)  # warm-up
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        T.tpmc_sweep_device(ctx, mesh, base, dd, None, K, N_each, out)
        b.record(stream)
        torch.cuda.synchronize(dev)
        ms = a.elapsed_time(b)
        res = T.results_from_bytes(out.cpu().numpy().tobytes(), K)
    finally:
        T.tpmc_mesh_unload(ctx, mesh)
    cm = {}
    for r, e, (al, be) in zip(res, E, grid):
        cm[(al, be)] = -float(np.dot(r["CM"], e))
    # trim angle per roll angle: the stable zero of C_m (falling through zero as alpha
    # grows) nearest alpha = 0, by linear interpolation
    trim = {}
    for be in betas:
        vals = [cm[(al, be)] for al in alphas]
        zeros = [alphas[k] + 10.0 * vals[k] / (vals[k] - vals[k + 1])
                 for k in range(len(alphas) - 1) if vals[k] >= 0.0 > vals[k + 1]]
        if zeros:
            trim[f"{be:g}"] = round(min(zeros, key=abs), 2)
    stable = all(cm[(al, be)] * al < 0.0 for (al, be) in grid if abs(al) >= 30.0)
    return {"workload": f"{case['name']}, chord 2 m, ref c/4, {K} attitudes x 2^22 particles, diffuse",
            "particles_per_s": K * N_each / (ms / 1e3), "ms": ms,
            "alpha_deg": alphas,
            "Cm_horizontal_m2": [round(cm[(al, 0.0)], 4) for al in alphas],
            "Cm_vertical_m2": [round(cm[(al, 90.0)], 4) for al in alphas],
            "trim_alpha_deg_by_beta": trim, "restoring_for_all_abs_alpha_ge_30": stable,
            "max_CD_sigma_rel": max(r["CD_sigma"] / r["CD"] for r in res)}


def measure_attitude_sweep(T, ctx, torch, stream, dev, ceil):
    """32 x 32 yaw/pitch grid x S in {5, 7.5, 10} on the satellite, 2^20 particles per
    item: one sweep call against 3,072 one-query calls (same N, so equal C_D
    error)."""
    case = W.satellite_case(N=1)
    grid = W.attitude_grid(32, 32)
    dirs = np.concatenate([grid] * 3)
    S = np.repeat([5.0, 7.5, 10.0], len(grid))
    K, N_each = len(S), 1 << 20
    mesh = T.tpmc_mesh_load(ctx, case["xyz"], case["tri"])
    try:
        base = T.make_params(**case["params"], stream_id=1 << 20)
        dd = torch.tensor(dirs, dtype=torch.float64, device=dev)
        ds = torch.tensor(S, dtype=torch.float64, device=dev)
        out = torch.zeros(K * T.RESULT_BYTES, dtype=torch.uint8, device=dev)
        T.tpmc_set_stream(ctx, stream)
        T.tpmc_sweep_device(ctx, mesh, base, dd[:64], ds[:64], 64, N_each, out)  # warm-up
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        T.tpmc_sweep_device(ctx, mesh, base, dd, ds, K, N_each, out)
        b.record(stream)
        torch.cuda.synchronize(dev)
        batched_ms = a.elapsed_time(b)
        res = T.results_from_bytes(out.cpu().numpy().tobytes(), K)
        T.tpmc_set_counters(ctx, True)
        T.tpmc_sweep_device(ctx, mesh, base, dd, ds, K, N_each, out)
        torch.cuda.synchronize(dev)
        T.tpmc_set_counters(ctx, False)
        res_c = T.results_from_bytes(out.cpu().numpy().tobytes(), K)
        assert all(x["sum_dv_q"] == y["sum_dv_q"] for x, y in zip(res, res_c))
        info = T.tpmc_mesh_info(ctx, mesh)
        roof = roofline_of([(work_of(res_c), info["node_bytes"], info["bvh_width"])], batched_ms / 1e3, ceil)
        T.tpmc_set_stream(ctx, None)
        c_mp = (2 * W.K_B * case["params"]["T_inf"] / case["params"]["m"]) ** 0.5
        t0 = time.perf_counter()
        same = 0
        for k in range(K):
            pk = dict(case["params"])
            pk["dir"] = tuple(dirs[k])
            pk["V"] = S[k] * c_mp
            r = T.tpmc_trace(ctx, mesh, T.make_params(**pk, stream_id=(1 << 20) + k), N_each)
            same += int(r["sum_dv_q"] == res[k]["sum_dv_q"])
        plain_s = time.perf_counter() - t0
        T.tpmc_set_stream(ctx, stream)
    finally:
        T.tpmc_mesh_unload(ctx, mesh)
    # the same launch with the schedule tpmc_tune picks on one 2^24-particle query,
    # in a context of its own so that the tuned schedule stays out of the other runs
    ctx2 = T.tpmc_create(0)
    try:
        T.tpmc_set_stream(ctx2, stream)
        mesh2 = T.tpmc_mesh_load(ctx2, case["xyz"], case["tri"])
        t0 = time.perf_counter()
        tuned = T.tpmc_tune(ctx2, mesh2, T.make_params(**case["params"]), 1 << 24)
        tune_s = time.perf_counter() - t0
        T.tpmc_sweep_device(ctx2, mesh2, base, dd[:64], ds[:64], 64, N_each, out)  # warm-up
        a.record(stream)
        T.tpmc_sweep_device(ctx2, mesh2, base, dd, ds, K, N_each, out)
        b.record(stream)
        torch.cuda.synchronize(dev)
        tuned_ms = a.elapsed_time(b)
        res2 = T.results_from_bytes(out.cpu().numpy().tobytes(), K)
        same_tuned = sum(int(x["sum_dv_q"] == y["sum_dv_q"]) for x, y in zip(res, res2))
    finally:
        T.tpmc_destroy(ctx2)
    n = K * N_each
    return {"workload": f"satellite 60,656 tri, 1,024 attitudes x S{{5,7.5,10}}, 2^20 particles each",
            "autotuned": {"particles_per_s": n / (tuned_ms / 1e3), "ms": tuned_ms, "launch": tuned,
                          "tune_s": tune_s, "items_bit_identical_to_untuned": same_tuned},
            "batched_particles_per_s": n / (batched_ms / 1e3), "batched_ms": batched_ms,
            "plain_particles_per_s": n / plain_s, "plain_ms": 1e3 * plain_s,
            "speedup_vs_plain": plain_s / (batched_ms / 1e3), "items_bit_identical_to_plain": same, "items": K,
            "roofline": roof,
            "median_CD_sigma_rel": float(np.median([r["CD_sigma"] / r["CD"] for r in res]))}


def measure_serving(T, ctx, rates=(100.0, 200.0, 400.0, 800.0), n_queries=1000):
    """Poisson streams of n_queries over four resident meshes (icosphere 1,280,
    cylinder 4,096, satellites 60k and 500k) at each arrival rate: continuous
    batching (submit/poll) against a server that runs one query per launch in
    arrival order, on the same arrival times and queries."""
    import threading as th

    ms = [M.icosphere(3), M.cylinder(), M.satellite(60_000), M.satellite(500_000)]
    ids = [T.tpmc_mesh_load(ctx, x, t) for x, t in ms]
    st = W.base_state()
    c_mp = (2 * W.K_B * st["T_inf"] / st["m"]) ** 0.5

    def params(q):
        return T.make_params(n=st["n"], T_inf=st["T_inf"], m=st["m"], V=q["S"] * c_mp, dir=q["dir"], T_W=st["T_W"],
                             eps_diffuse=0.9, A_ref=1.0, seed=q["seed"], max_bounces=64)

    out = {}
    try:
        warm = W.serving_stream(1, 100.0, seed=3)[0]
        for i in ids:  # warm-up per mesh, through both paths
            T.tpmc_trace(ctx, i, params(warm), 100_000)
            T.tpmc_poll(ctx, T.tpmc_submit(ctx, i, params(warm), 100_000), -1)
        for rate in rates:
            stream = W.serving_stream(n_queries, rate, seed=3)
            # continuous batching
            handles = [None] * len(stream)
            t_start = time.perf_counter() + 0.05

            def submitter():
                for k, q in enumerate(stream):
                    d = t_start + q["t_arrival"] - time.perf_counter()
                    if d > 0:
                        time.sleep(d)
                    handles[k] = T.tpmc_submit(ctx, ids[q["mesh"]], params(q), q["N"])

            thr = th.Thread(target=submitter)
            thr.start()
            thr.join()
            lat = [T.tpmc_poll(ctx, h, -1)["ms"] for h in handles]
            cb_span = time.perf_counter() - t_start
            # one query per launch, first come first served
            t_start = time.perf_counter() + 0.05
            lat_plain = []
            for q in stream:
                d = t_start + q["t_arrival"] - time.perf_counter()
                if d > 0:
                    time.sleep(d)
                T.tpmc_trace(ctx, ids[q["mesh"]], params(q), q["N"])
                lat_plain.append(1e3 * (time.perf_counter() - (t_start + q["t_arrival"])))
            plain_span = time.perf_counter() - t_start
            n = sum(q["N"] for q in stream)
            out[f"{rate:g}"] = {
                "workload": f"{n_queries} Poisson queries at {rate:g}/s, N log-uniform [1e5,1e8], S~U[3,12], "
                            "4 resident meshes (1,280 / 4,096 / 60,656 / 503,537 tri)",
                "p50_ms": float(np.percentile(lat, 50)), "p99_ms": float(np.percentile(lat, 99)),
                "throughput_particles_per_s": n / cb_span,
                "plain": {"p50_ms": float(np.percentile(lat_plain, 50)), "p99_ms": float(np.percentile(lat_plain, 99)),
                          "throughput_particles_per_s": n / plain_span}}
    finally:
        for i in ids:
            T.tpmc_mesh_unload(ctx, i)
    return out


# ---------------------------------------------------------------- GPU side
def run_ours(args):
    import torch

    from paper_1312_3691_gb300 import tpmc as T
    from paper_1312_3691_gb300.build import build

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    dist = None
    if world > 1:
        import torch.distributed as dist_mod

        dist = dist_mod
        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
    if rank == 0:
        build()
    if dist is not None:
        dist.barrier()
    build()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    props = torch.cuda.get_device_properties(dev)
    ctx = T.tpmc_create(local)
    # a dedicated stream: the library launches on it and the CUDA events are recorded on it
    stream = torch.cuda.Stream(dev)
    torch.cuda.set_stream(stream)
    T.tpmc_set_stream(ctx, stream)
    gs = groups()
    K = len(gs[0]["cases"])
    mesh_ids = {}
    for g in gs:
        if g["shape"] not in mesh_ids:
            mesh_ids[g["shape"]] = T.tpmc_mesh_load(ctx, g["xyz"], g["tri"])
    d_in = []
    for gi, g in enumerate(gs):
        # ranks trace independent streams of the same workload (weak scaling)
        base = T.make_params(**g["base"], stream_id=rank_stream_base(rank, gi))
        d_in.append((mesh_ids[g["shape"]], base,
                     torch.tensor(g["dirs"], dtype=torch.float64, device=dev),
                     torch.tensor(g["S"], dtype=torch.float64, device=dev),
                     torch.zeros(K * T.RESULT_BYTES, dtype=torch.uint8, device=dev)))
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)

    def step(events=None):
        for i, (mid, base, dd, ds, out) in enumerate(d_in):
            if events is not None:
                events[i][0].record(stream)
            T.tpmc_sweep_device(ctx, mid, base, dd, ds, K, N_EACH, out)
            if events is not None:
                events[i][1].record(stream)

    # counters pass (outside timing): algorithmic work per step
    T.tpmc_set_counters(ctx, True)
    step()
    torch.cuda.synchronize(dev)
    T.tpmc_set_counters(ctx, False)
    group_work = []
    for (_, _, _, _, out) in d_in:
        res = T.results_from_bytes(out.cpu().numpy().tobytes(), K)
        assert all(r["status"] == 0 for r in res), res
        group_work.append(work_of(res))
    work = work_of([])
    for w in group_work:
        for k in work:
            work[k] += w[k]
    mesh_info = {shape: T.tpmc_mesh_info(ctx, mid) for shape, mid in mesh_ids.items()}

    for _ in range(args.warmup):
        flush.zero_()
        step()
    torch.cuda.synchronize(dev)
    if dist is not None:
        dist.barrier()
    torch.cuda.synchronize(dev)
    uuid = str(getattr(props, "uuid", "") or "")
    sampler = ClockSampler(uuid if uuid.startswith("GPU-") else (f"GPU-{uuid}" if uuid else local))
    sampler.start()
    time.sleep(0.3)
    step_ms, launch_ms = [], []
    for _ in range(args.steps):
        flush.zero_()
        ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in d_in]
        step(ev)
        torch.cuda.synchronize(dev)
        ms = [a.elapsed_time(b) for a, b in ev]
        launch_ms += ms
        step_ms.append(sum(ms))
    torch.cuda.synchronize(dev)
    clocks = sampler.stop()
    t_step = max_over_ranks(sum(step_ms) / len(step_ms), dist, dev)
    particles_step = work["particles"]
    value = world * particles_step / (t_step / 1e3)

    # results of the last timed step
    results_by_group = [T.results_from_bytes(out.cpu().numpy().tobytes(), K) for (*_, out) in d_in]

    # end to end through the public API with host buffers
    e2e_ms = []
    h2d = d2h = 0
    T.tpmc_set_stream(ctx, None)
    for k in range(max(1, args.e2e_steps)):
        flush.zero_()
        torch.cuda.synchronize(dev)
        t0 = time.perf_counter()
        ids = {}
        h2d = d2h = 0
        for g in gs:
            if g["shape"] not in ids:
                ids[g["shape"]] = T.tpmc_mesh_load(ctx, g["xyz"], g["tri"])
                h2d += T.tpmc_mesh_info(ctx, ids[g["shape"]])["device_bytes"]
            base = T.make_params(**g["base"], stream_id=rank * 4096 + 7)
            res = T.tpmc_sweep(ctx, ids[g["shape"]], base, g["dirs"], g["S"], N_EACH)
            h2d += g["dirs"].nbytes + g["S"].nbytes
            d2h += len(res) * T.RESULT_BYTES
        for i in ids.values():
            T.tpmc_mesh_unload(ctx, i)
        e2e_ms.append(1e3 * (time.perf_counter() - t0))
    e2e_t = max_over_ranks(statistics.mean(e2e_ms), dist, dev)
    e2e_value = world * particles_step / (e2e_t / 1e3)

    peaks = measured_peaks()
    sm_max = float(peaks.get("sm_max_mhz", 2070.0))
    alu_peak_tflops = props.multi_processor_count * FP32_LANES_PER_SM * 2 * sm_max * 1e6 / 1e12
    traffic = TRACE_TRAFFIC.get(kernel_source_hash())
    # measured ceilings: particles/s <= min(L2 rate / bytes per particle, FP32 rate / flops per particle)
    ceil = T.tpmc_measure_ceilings(ctx)
    mean_step_s = statistics.mean(step_ms) / 1e3
    parts = [(w, mesh_info[g["shape"]]["node_bytes"], mesh_info[g["shape"]]["bvh_width"])
             for w, g in zip(group_work, gs)]
    roof = roofline_of(parts, mean_step_s, ceil)
    roof.update({"traffic": traffic, "kernel": "seed_kernel<float> and trace_kernel<float>, all batches of a sweep call",
                 "achieved_definition": "algorithmic L2 bytes (node and triangle reads) per sweep call / mean duration "
                                        "of a call (CUDA events on the launching stream)",
                 "launch_ms_mean": statistics.mean(launch_ms),
                 "fp32_alu_derived_tflops": alu_peak_tflops,
                 "fp32_alu_basis": f"{props.multi_processor_count} SMs x {FP32_LANES_PER_SM} FP32 lanes x 2 (FMA) x "
                                   f"{sm_max:.0f} MHz (sm_max_mhz of MEASURED_PEAKS.json)"})
    extras = {}
    if rank == 0 and not args.no_extras:
        extras["satellite"] = measure_satellite(T, ctx, torch, stream, ceil)
        extras["satellite_500k"] = measure_satellite(T, ctx, torch, stream, ceil, target_triangles=500_000)
        extras["concave_hemisphere"] = measure_hemisphere(T, ctx)
        extras["box_cv"] = measure_box_cv(T, ctx)
        extras["moment_sweep"] = measure_moment_sweep(T, ctx, torch, stream, dev)
        extras["attitude_sweep"] = measure_attitude_sweep(T, ctx, torch, stream, dev, ceil)
        extras["serving_by_rate"] = measure_serving(T, ctx)
        extras["serving"] = extras["serving_by_rate"]["100"]
    if rank == 0:
        cpu_base, cd_err, cd_other, parity = (None, None, None, None)
        if not args.no_cpu_baseline:
            cpu_base, cd_err, cd_other, parity = cpu_baseline_leg(T, ctx, results_by_group)
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": t_step, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32",
            "data": "synthetic (procedural meshes; paper prints no absolute throughput)",
            "config": {"workload": WORKLOAD, "particles_per_step": particles_step, "cases": 4 * K,
                       "sweep_calls_per_step": len(d_in), "l2": "256 MiB flush between steps, outside timed intervals",
                       "precision": "FP32 traversal, FP64 set-up and reduction"},
            "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(d2h),
                    "ms_per_step": e2e_t, "includes": "mesh upload + BVH build, host inputs, host results"},
            "gpu_launches": args.steps * len(d_in) * launches_per_call(len(gs[0]["dirs"]) * N_EACH),
            "roofline": roof,
            "clocks": clocks,
            "cpu_baseline": cpu_base,
            "cd_error": cd_err, "cd_error_other_configs": cd_other, "parity": parity,
            "serve": {k: extras["serving"][k] for k in ("p50_ms", "p99_ms", "throughput_particles_per_s", "plain")}
            if "serving" in extras else None,
            "extras": extras,
        }
        print(json.dumps(line), flush=True)
    T.tpmc_destroy(ctx)
    if dist is not None:
        dist.destroy_process_group()
    return 0


def run_profile_launch(args):
    """One warm-up and one measured sweep launch of one group of the workload at a
    reduced particle count, for profiler captures (ncu -k "regex:(seed|trace)_kernel": a pair per batch of 2^26)."""
    import torch

    from paper_1312_3691_gb300 import tpmc as T
    from paper_1312_3691_gb300.build import build

    build()
    if args.profile_launch in ("satellite-sweep", "satellite500k-sweep"):
        case = W.satellite_case(N=1, target_triangles=500_000 if "500k" in args.profile_launch else 60_000)
        grid = W.attitude_grid(8, 12)
        g = {"xyz": case["xyz"], "tri": case["tri"], "base": case["params"], "dirs": grid,
             "S": np.full(len(grid), 7.0), "cases": list(range(len(grid)))}
    else:
        shape, gsi = args.profile_launch.split("-")
        g = [x for x in groups() if x["shape"] == shape and x["eps"] == (1.0 if gsi == "diffuse" else 0.0)][0]
    ctx = T.tpmc_create(0)
    stream = torch.cuda.Stream()
    torch.cuda.set_stream(stream)
    T.tpmc_set_stream(ctx, stream)
    if args.launch:
        vals = [int(x) for x in args.launch.split(",")] + [0, 0, 0]
        T.tpmc_set_launch(ctx, block=vals[0], blocks_per_sm=vals[1], chunk=vals[2], smem_nodes=vals[3],
                          refill_at=vals[4], bvh_leaf=vals[5], bvh_width=vals[6])
    mesh = T.tpmc_mesh_load(ctx, g["xyz"], g["tri"])
    K = len(g["cases"])
    dd = torch.tensor(g["dirs"], dtype=torch.float64, device="cuda")
    ds = torch.tensor(g["S"], dtype=torch.float64, device="cuda")
    out = torch.zeros(K * T.RESULT_BYTES, dtype=torch.uint8, device="cuda")
    base = T.make_params(**g["base"])
    times = []
    for _ in range(2):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        T.tpmc_sweep_device(ctx, mesh, base, dd, ds, K, args.profile_n_each, out)
        b.record(stream)
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    res = T.results_from_bytes(out.cpu().numpy().tobytes(), K)
    assert all(r["status"] == 0 for r in res)
    n = K * args.profile_n_each
    print(json.dumps({"profile_launch": args.profile_launch, "particles": n, "ms": times[-1],
                      "particles_per_s": n / (times[-1] / 1e3), "launch": T.tpmc_get_launch(ctx, mesh)}))
    T.tpmc_destroy(ctx)
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--e2e-steps", type=int, default=2)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-extras", action="store_true", help="skip the satellite, attitude-sweep and serving runs")
    ap.add_argument("--profile-launch", default=None,
                    help="plate-specular|plate-diffuse|cylinder-specular|cylinder-diffuse|satellite-sweep|"
                         "satellite500k-sweep: one small launch")
    ap.add_argument("--profile-n-each", type=int, default=100_000)
    ap.add_argument("--launch", default=None,
                    help="block,blocks_per_sm,chunk,smem_nodes[,refill_at,bvh_leaf,bvh_width] for --profile-launch "
                         "(block 0: only the BVH layout)")
    args = ap.parse_args()
    if args.profile_launch:
        return run_profile_launch(args)
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
