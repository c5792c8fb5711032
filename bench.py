#!/usr/bin/env python3
"""Pressure solves/s + Ginteractions/s on the 2048^2 rigid-cylinder snapshot.

One step = the whole path on one synthetic snapshot, inputs resident in HBM:
  pp_rhs (Poisson source + leaf multipoles) -> pp_pressure_solve (upward pass,
  multipole-to-local/local-to-local, local evaluation + near field, pressure at
  all n^2 cells) -> pp_surface_traction (tree-code pressure at the surface points,
  tractions, FP64 drag/lift).
Default workload: cylinder D = 0.1 at (0.3, 0.5) on 2048^2 cells, potential flow +
64-blob wake, lambda = 1e4, nu = 1e-4, mixed precision with the order, theta and near-field
tile the autotuner picks for this snapshot under the 1e-4 error bound (--no-autotune keeps
--order/--theta/--tile), 2048 surface points lifted by 2h.  L2 is flushed (a 256 MB write)
between timed steps.  The step is replayed as one CUDA graph.

Prints ONE JSON line (rank 0).  Under torchrun each rank solves its own snapshots
(independent problems: weak scaling, no collective in the data path).
``--impl reference`` times the CPU oracle on a bounded sample of the same workload.

Besides the headline keys the line carries: ``roofline`` (the dominant stage against its
peak, with its DRAM traffic from profiles/ncu_traffic.txt), ``stages`` and ``stage_timing``
(per-stage event times from a second pass), ``e2e`` (the same metric from pinned host
memory through pp_pipeline), ``serve`` (the pp_server latency and throughput runs),
``penal_force`` (the penalisation-force reduction, Eq. dragPenal), ``fft_solve`` (the
zero-padded FFT solve of the same discrete sum beside the multipole grid solve),
``adaptive_solve`` (the FP64 solve on an adaptive grid refined towards the cylinder),
``cpu_baseline`` (the oracle on the host cores) and ``clocks``.
"""
import argparse
import hashlib
import json
import math
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "pressure solves/s + Ginteractions/s at 2048² grid; p50/p99 serve latency"
L2_FLUSH_BYTES = 256 << 20


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=None,
                    help="timed steps (default: 2000 for our arm, about half a second of GPU time, so the "
                         "clock samples fall inside it; 10 for the CPU reference arm)")
    ap.add_argument("--warmup", type=int, default=None, help="untimed warm-up steps (default 20; 3 reference)")
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--n", type=int, default=2048)
    ap.add_argument("--precision", default="mixed", choices=["mixed", "fp64"])
    ap.add_argument("--order", type=int, default=20)
    ap.add_argument("--theta", type=float, default=0.5)
    ap.add_argument("--npts", type=int, default=2048)
    ap.add_argument("--tile", type=int, default=16, choices=[8, 16, 128])
    ap.add_argument("--theta-surface", type=float, default=0.0,
                    help="surface tree-code acceptance (0: min(theta, 0.6)); autotuned by default")
    ap.add_argument("--m2l-tensor", action="store_true",
                    help="mixed plans: the multipole-to-local translations on the tensor cores")
    ap.add_argument("--no-autotune", action="store_true",
                    help="mixed path: keep --order/--theta/--tile instead of the autotuned setting")
    ap.add_argument("--no-serve", action="store_true", help="skip the short serving measurement")
    ap.add_argument("--serve-sweep", action="store_true",
                    help="serving workload only: 2000 requests per rate, grids 256^2-4096^2, rates 50-2000/s")
    ap.add_argument("--serve-requests", type=int, default=2000, help="requests per serving rate")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-batch", action="store_true", help="skip the 64-snapshot swimmer batch measurement")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-targets", type=int, default=2048,
                    help="grid targets of the oracle's bounded CPU sample")
    return ap.parse_args()


def dist_env():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


def workload_config(a):
    return {"workload": f"cylinder_{a.n}x{a.n}_{a.precision}", "grid": a.n, "order": a.order,
            "theta": a.theta, "tile": a.tile, "theta_surface": a.theta_surface or min(a.theta, 0.6),
            "m2l": "tensor" if getattr(a, "m2l_tensor", False) else "fp32",
            "leaf_cells": 64, "surface_points": a.npts, "lambda": 1e4,
            "nu": 1e-4, "lift": "2h", "l2": "flushed between steps (256 MB write)", "seed": 2000}


# ----------------------------------------------------------------------------- clocks
class ClockSampler:
    """nvidia-smi sampled every 50 ms during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.path = None

    def start(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "50"],
                                         stdout=self.f, stderr=subprocess.DEVNULL)
            time.sleep(0.1)  # the first sample lands before the timed region starts
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        time.sleep(0.25)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.f.close()
        sm, smax, reasons = [], 0, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax = max(smax, float(parts[2]))
            except ValueError:
                continue
            for nm, val in zip(names, parts[5:9]):
                if val.lower().startswith("active"):
                    reasons.add(nm)
        os.unlink(self.path)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": smax, "reasons": sorted(reasons),
                "samples": len(sm)}


# ------------------------------------------------------------------------ roofline
def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        try:
            return json.load(open(p)), "measured"
        except Exception:
            pass
    return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0}, "fallback"


def fp32_peak_tflops(n_sm):
    """FP32 FMA nominal: SMs x 128 FP32 lanes x 2 flops x 2.07 GHz (maximum SM clock); used
    only when the measurement below fails."""
    return n_sm * 128 * 2 * 2.07e9 / 1e12


def fp64_peak_tflops():
    """GB300 FP64 nominal (the part's non-tensor FP64 rate); used only when the measurement fails."""
    return 1.25


_ALU = {}


def alu_peaks(local=0):
    """FP32 FMA, special-function lg2 and FP64 FMA throughput measured on this GPU by
    pp_measure_alu_peaks (independent chains of one instruction filling every SM; best of 30
    launches of 1-3 ms each), with nvidia-smi clocks sampled during the measurement and the
    per-SM per-clock rates they imply.  Cached for the process."""
    if "v" in _ALU:
        return _ALU["v"]
    from paper_1610_04398_gb300 import api
    clocks = ClockSampler(local)
    clocks.start()
    try:
        pk = api.measure_alu_peaks(reps=30)
    except Exception as e:  # reported, and the roofline falls back to the nominal figures
        pk = {"error": f"{type(e).__name__}: {e}"}
    clk = clocks.stop()
    pk["clocks"] = clk
    if clk and "fp32_tflops" in pk:
        f = clk["sm_mhz"] * 1e6 * pk["sms"]
        pk["per_sm_per_clock"] = {"fp32_fma": pk["fp32_tflops"] * 1e12 / 2 / f, "lg2": pk["lg2_gops"] * 1e9 / f,
                                  "fp64_fma": pk["fp64_tflops"] * 1e12 / 2 / f}
    _ALU["v"] = pk
    return pk


def alu_peak(precision, n_sm, local=0):
    """(peak TFLOP/s, source) for the ALU roofline of a plan precision."""
    pk = alu_peaks(local)
    key = "fp32_tflops" if precision == "mixed" else "fp64_tflops"
    if key in pk:
        return pk[key], f"measured by pp_measure_alu_peaks ({'FP32' if precision == 'mixed' else 'FP64'} FMA chains)"
    if precision == "mixed":
        return fp32_peak_tflops(n_sm), "nominal FP32: SMs x 128 lanes x 2 flops x 2.07 GHz (measurement failed)"
    return fp64_peak_tflops(), "nominal FP64 1.25 TFLOP/s (measurement failed)"


def fixed_peak(n_sm, local=0):
    """(peak TFLOP/s, source) of FP64 sums in fixed point: 32 x 32 + 64 bit integer multiply-adds at the
    28 lanes a clock and SM measured on GB300, three in place of a fused multiply-add (2 flops)."""
    pk = alu_peaks(local)
    mhz = (pk.get("clocks") or {}).get("sm_mhz") or 2070.0
    return 2 * 28 / 3 * pk.get("sms", n_sm) * mhz * 1e6 / 1e12, \
        "integer multiply-adds, 28 lanes a clock and SM measured, three a product"


# The sources that build and launch each kernel a traffic record covers (its header, the
# translation units that instantiate it, the C ABI that sizes its launches).
_STEP_SOURCES = ("pp_common.h", "pp_kernels.cuh", "pp_fast.cuh", "pp_fp64.cuh", "pp_fixed.cuh",
                 "pp_log.cuh", "pp_surface.cuh", "pp_kernels_f32.cu", "pp_kernels_f64.cu",
                 "pp_tc.cu", "pp_tcgen05.cuh", "pp_capi.cu")
KERNEL_SOURCES = {"k_m2l_reg": _STEP_SOURCES, "k_m2l_far": _STEP_SOURCES, "k_m2l_tc": _STEP_SOURCES + ("pp_m2l_tc.cu",),
                  "k_near_tc": _STEP_SOURCES,
                  "k_fft_solve": ("pp_common.h", "pp_fft.cu", "pp_capi.cu")}


def kernel_src_hash(kernel="k_m2l_reg"):
    h = hashlib.sha256()
    d = os.path.join(ROOT, "paper_1610_04398_gb300", "csrc")
    for fn in sorted(set(KERNEL_SOURCES.get(kernel, _STEP_SOURCES))):
        h.update(open(os.path.join(d, fn), "rb").read())
    return h.hexdigest()[:16]


def recorded_traffic(kernel, workload):
    """dram bytes per launch from profiles/ncu_traffic.txt, if taken on the kernel's current source."""
    p = os.path.join(ROOT, "profiles", "ncu_traffic.txt")
    if not os.path.exists(p):
        return None
    src = kernel_src_hash(kernel)
    for line in open(p):
        if line.startswith("#") or not line.strip():
            continue
        kv = dict(x.split("=", 1) for x in line.split() if "=" in x)
        if kv.get("kernel") == kernel and kv.get("workload") == workload and kv.get("src") == src:
            return float(kv["dram_bytes_per_launch"])
    return None


def m2l_flops(P1):
    """Flops of one factored multipole-to-local translation (diag * real R * diag):
    x_k = tau^-k M_k (6 per complex product), row 0 real (2 per term), rows l >= 1
    (4 per term: re and im FMAs, plus the monopole column), output tau^-l y_l added to L_l (8)."""
    p = P1 - 1
    return 6 * p + 2 * p + p * (4 * p + 2) + 8 * p


def shift_flops(P1):
    """Flops of one factored M2M or L2L shift: two complex diagonals and a triangular real product."""
    p = P1 - 1
    return 12 * p + 4 * p * (p + 1) // 2


def stage_work(info, n, P1, prec_bytes, fused_leaf):
    """Algorithmic work of each stage of one step (flops or bytes).  With ``fused_leaf``
    (the mixed path's split solve) the leaf stage is the near field alone and the leaf_m2l
    stage runs after it: with the two-launch downward pass (info.downward == 2) the
    downward stage is every level's multipole-to-local translations and leaf_m2l the
    local-to-local shifts plus the local evaluation; otherwise the downward stage holds the
    translations and shifts of every level and leaf_m2l the evaluation alone."""
    L = info.levels - 1
    nbox = (4 ** (L + 1) - 1) // 3
    nleaf = 4 ** L
    l2p = n * n * (P1 - 1) * 8.0          # p complex Horner steps (8 flops) per cell
    near = info.near_pairs * 2.0          # one FMA per source/target pair
    m2l = info.m2l_pairs * m2l_flops(P1)
    l2l = (nbox - 21) * shift_flops(P1)   # one shift into every box of levels 3..L
    two = fused_leaf and (prec_bytes == 8 or getattr(info, "downward", 0) >= 2)  # FP64: k_m2l64, then k_down64
    return {
        # RHS: read u, v, chi, us_x, us_y, write q (plan precision)
        "rhs_p2m": ("hbm", 6.0 * n * n * prec_bytes),
        "upward": ("alu", (nbox - nleaf) * 4 * shift_flops(P1)),
        "downward": ("alu", m2l if two else m2l + l2l),
        "leaf": ("alu", near if fused_leaf else near + l2p),
        "leaf_m2l": ("alu", (l2l + l2p if two else l2p) if fused_leaf else None),
        "surface": ("latency", None),
    }


# ----------------------------------------------------------------------- our arm
def run_ours(a):
    import torch
    import torch.distributed as dist
    from paper_1610_04398_gb300 import api, synth

    rank, world, local = dist_env()
    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    import paper_1610_04398_gb300 as pkg
    if rank == 0:
        pkg.build()
    if world > 1:
        dist.barrier()
    # independent problems per rank (weak scaling): rank r solves the snapshot of seed 2000 + r
    snap = synth.cylinder_flow(a.n, seed=2000 + rank, n_surface=a.npts)
    tuned = None
    if a.precision == "mixed" and not a.no_autotune:
        from paper_1610_04398_gb300 import autotune
        tuned = autotune.autotune(snap, steps=5)
        a.order, a.theta, a.tile = tuned["best"]["order"], tuned["best"]["theta"], tuned["best"]["tile"]
        a.theta_surface = tuned["best"]["theta_surface"]
    plan = api.Plan(a.n, snap.h, a.order, a.theta, precision=a.precision, lift=snap.lift, uinf=snap.uinf,
                    tile=a.tile, theta_surface=a.theta_surface, m2l_tensor=a.m2l_tensor)
    dt = plan.dtype
    host = [torch.from_numpy(np.ascontiguousarray(x)).to(dt) for x in
            (snap.u, snap.v, snap.chi, snap.usx, snap.usy)]
    dev = [x.cuda() for x in host]
    pts = torch.from_numpy(snap.points).cuda()
    nrm = torch.from_numpy(snap.normals).cuda()
    P = torch.empty(a.n * a.n, dtype=dt, device="cuda")
    F = torch.zeros(6, dtype=torch.float64, device="cuda")
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.float32, device="cuda")

    # the whole step is one CUDA graph (pp_step_graph_create), replayed every step.  The
    # headline steps replay the plain graph; the per-stage durations come from a second
    # pass of equal length over a copy captured with stage events (the event nodes
    # themselves cost ~10% of a 2048^2 step, so they stay out of the headline timing).
    plan.enable_timing(False)
    graph = plan.capture_step(*dev, snap.lam, p_out=P, points=pts, normals=nrm, nu=snap.nu, forces=F)
    plan.enable_timing(True)
    graph_t = plan.capture_step(*dev, snap.lam, p_out=P, points=pts, normals=nrm, nu=snap.nu, forces=F)

    for _ in range(max(a.warmup, 3)):
        graph.launch()
    torch.cuda.synchronize()
    stream = torch.cuda.current_stream()
    stage_ms = {k: [] for k in api.Plan.STAGES}
    step_ms = []
    clocks = ClockSampler(local)
    launches0 = plan.info().launches
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    clocks.start()
    wall0 = time.perf_counter()
    # every step is queued before the GPU reaches it (a GPU-side sleep lets the host run
    # ahead), so each event pair brackets the step's device work only, not host launch gaps
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(a.steps)]
    torch.cuda._sleep(int(min(2e9, 1.2e5 * a.steps)))
    for e0, e1 in ev:
        flush.zero_()
        e0.record(stream)
        graph.launch()
        e1.record(stream)
    torch.cuda.synchronize()
    step_ms = [e0.elapsed_time(e1) for e0, e1 in ev]
    wall = time.perf_counter() - wall0
    clk = clocks.stop()
    launches = plan.info().launches - launches0
    tot_s = sum(step_ms) / 1e3
    if world > 1:
        t = torch.tensor([tot_s], device="cuda", dtype=torch.float64)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        tot_s = float(t.item())
    # stage pass: the same number of steps over the graph with stage events
    for _ in range(3):
        graph_t.launch()
    torch.cuda.synchronize()
    stage_step_ms = []
    for _ in range(a.steps):
        flush.zero_()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        graph_t.launch()
        e1.record(stream)
        st = plan.stage_times()  # waits for the step's last stage event
        e1.synchronize()
        stage_step_ms.append(e0.elapsed_time(e1))
        for k, v in st.items():
            stage_ms[k].append(v)
    graph_t.destroy()
    plan.enable_timing(False)
    info = plan.info()

    value = a.steps * world / tot_s
    ms_per_step = tot_s * 1e3 / a.steps
    ginter = info.near_pairs * a.steps * world / tot_s / 1e9
    P1 = a.order + 1
    prec_bytes = 4 if a.precision == "mixed" else 8
    fused = bool(stage_ms["leaf_m2l"]) and stage_ms["leaf_m2l"][0] >= 0
    work = stage_work(info, a.n, P1, prec_bytes, fused)
    props = torch.cuda.get_device_properties(local)
    peaks, peak_src = measured_peaks()
    alu_pk, alu_src = alu_peak(a.precision, props.multi_processor_count, local)
    stages = {}
    for k, vals in stage_ms.items():
        ms = statistics.mean(vals) if vals and vals[0] >= 0 else None
        bound, amount = work[k]
        ent = {"ms": ms, "bound": bound}
        if ms and amount:
            if bound == "hbm":
                ent["achieved_gbs"] = amount / (ms / 1e3) / 1e9
                ent["frac"] = ent["achieved_gbs"] / peaks["hbm_gbs"]
            else:
                ent["achieved_tflops"] = amount / (ms / 1e3) / 1e12
                ent["frac"] = ent["achieved_tflops"] / alu_pk
        stages[k] = ent
    # the roofline is reported for the longest stage whose algorithmic work is defined
    # (the surface stage is a latency-bound tree walk with no such figure)
    dom = max((k for k in stages if stages[k]["ms"] and work[k][1]), key=lambda k: stages[k]["ms"])
    f64 = a.precision == "fp64" and a.order <= 23 and info.levels > 2  # the fixed-point kernels
    near_name = {128: "k_near_tc", 16: "k_near16", 8: "k_leaf_fast"}.get(info.near_kernel, "k_near64" if f64 else "k_leaf")
    if info.near_kernel == 128 and stages["leaf"]["ms"]:
        # the near field is a dense contraction on the tensor cores (kind::f16, FP32
        # accumulate): its roofline is the dense FP16 tensor peak, which is the measured
        # bf16 peak (the two rates are equal); three FP16 products per FP32-accurate term
        # cap frac at 1/3
        e = stages["leaf"]
        e["bound"] = "tensor"
        e["peak_tflops"] = peaks["bf16_tflops"]
        e["frac"] = e["achieved_tflops"] / e["peak_tflops"]
    two = fused and info.downward >= 2
    far = "k_m2l_tc" if info.downward == 3 else "k_m2l_far"
    kern = {"leaf": near_name if fused else "k_leaf", "downward": far if two else "k_m2l64" if f64 else "k_m2l_reg",
            "rhs_p2m": "k_rhs64" if f64 else "k_rhs_p2m_fast",
            "upward": "k_up_tree" if a.precision == "mixed" else "k_up64" if f64 else "k_m2m_reg",
            "leaf_m2l": "k_down_tree" if two else "k_down64" if f64 else "k_l2p_leaf", "surface": "k_surface"}[dom]
    d = stages[dom]
    if d["bound"] == "tensor":
        roof = {"bound": "tensor", "achieved": d["achieved_tflops"], "peak": d["peak_tflops"], "unit": "TFLOP/s",
                "frac": d["frac"],
                "peak_source": f"{peak_src} bf16_tflops (= the dense FP16 rate); the 3-product FP16 split caps frac at 1/3"}
    elif d["bound"] == "hbm":
        roof = {"bound": "hbm", "achieved": d["achieved_gbs"], "peak": peaks["hbm_gbs"], "unit": "GB/s",
                "frac": d["frac"], "peak_source": f"{peak_src} hbm_gbs"}
    else:
        roof = {"bound": "alu", "achieved": d.get("achieved_tflops"), "peak": alu_pk, "unit": "TFLOP/s",
                "frac": d.get("frac"), "peak_source": alu_src}
        if f64 and dom in ("leaf", "downward") and roof["achieved"]:
            roof["peak"], roof["peak_source"] = fixed_peak(props.multi_processor_count, local)
            roof["frac"] = roof["achieved"] / roof["peak"]
    roof["kernel"] = kern
    roof["concurrent"] = fused  # the near field shares the GPU with the expansion passes
    alu_total = sum(w[1] for k, w in work.items() if w[0] == "alu" and w[1])
    roof["step_alu_frac"] = alu_total / (ms_per_step / 1e3) / 1e12 / alu_pk
    tr = recorded_traffic(kern, workload_config(a)["workload"])
    roof["traffic"] = tr
    lat = sorted(step_ms)
    out = {
        "metric": METRIC, "value": value, "unit": "solves/s", "n_gpus": world, "steps": a.steps,
        "warmup": a.warmup, "ms_per_step": ms_per_step, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32+f64" if a.precision == "mixed" else "f64", "data": "synthetic",
        "config": workload_config(a),
        "ginteractions_per_s": ginter,
        "ginteractions_effective_per_s": (a.n * a.n + a.npts) * a.n * a.n * a.steps * world / tot_s / 1e9,
        "ginteractions_note": ("ginteractions_per_s: near-field cell pairs of the grid solve per second (the surface "
                               "tree-code's leaf pairs are not counted); effective: the direct-sum equivalent, "
                               "(n^2 + surface points) x n^2 pairs per solve"),
        "latency_ms": {"p50": lat[len(lat) // 2], "p99": lat[min(len(lat) - 1, int(0.99 * len(lat)))]},
        "roofline": roof, "stages": stages,
        "stage_timing": {"pass": "second run of the same steps over the step graph captured with stage events",
                         "ms_per_step": statistics.mean(stage_step_ms)},
        "near_kernel": near_name, "gpu_launches": int(launches),
        "clocks": clk, "wall_s": wall,
    }
    if tuned is not None:
        nominal = [r for r in tuned["table"] if r["order"] == 20 and r["theta"] == 0.5 and r["stage"] == 1]
        out["autotune"] = {"best": tuned["best"], "reference": tuned["reference"], "tol": tuned["tol"],
                           "safety": tuned["safety"], "candidates": len(tuned["table"]),
                           "seconds": round(tuned["seconds"], 2),
                           "p20_theta05": nominal,
                           "table_columns": TUNE_COLUMNS, "table": tune_table(tuned)}
    out["alu_peaks"] = alu_peaks(local)
    if tuned is not None:
        out["in_config"] = in_config_measure(a, tuned, snap, dev, pts, nrm, flush)
    out["penal_force"] = penal_measure(a, plan, dev, snap, F, peaks)
    if a.n <= 4096:
        out["fft_solve"] = fft_measure(a, plan, peaks)
    try:
        out["adaptive_solve"] = adaptive_measure()
    except Exception as e:  # the adaptive path is reported, never allowed to stop the bench line
        out["adaptive_solve"] = {"error": f"{type(e).__name__}: {e}"}
    setting = None
    if (not a.no_batch or not a.no_serve) and world == 1:
        try:
            t0 = time.perf_counter()
            synth.set_device("cuda")
            try:
                swimmers = synth.swimmer_batch(64)
            finally:
                synth.set_device(None)
            t_synth = time.perf_counter() - t0
            setting, tune_info = swimmer_setting(swimmers)
            out["swimmer_setting"] = dict(tune_info, synth_s=t_synth)
            if not a.no_batch:
                out["swimmer_batch"] = batch_measure(a, flush, swimmers, setting)
            del swimmers
        except Exception as e:  # reported, never allowed to stop the bench line
            out["swimmer_batch"] = {"error": f"{type(e).__name__}: {e}"}
    if not a.no_e2e:
        graph.destroy()
        out["e2e"] = e2e(a, plan, snap, host, world)
    if not a.no_serve and world == 1:
        out["serve"] = serve_summary(a, requests=a.serve_requests, setting=setting)
        out["latency_ms"]["serve_p50"] = out["serve"]["poisson_1000"]["p50_ms"]
        out["latency_ms"]["serve_p99"] = out["serve"]["poisson_1000"]["p99_ms"]
    if rank == 0 and world == 1 and not a.no_cpu_baseline:
        out["cpu_baseline"] = cpu_baseline(a, snap)
    if rank == 0:
        print(json.dumps(out), flush=True)
    graph.destroy()
    plan.destroy()
    if world > 1:
        dist.barrier()
        dist.destroy_process_group()


TUNE_COLUMNS = ["order", "theta", "tile", "theta_surface", "ms", "err_p", "worst_p", "err_surface",
                "worst_surface", "err_force"]


def tune_table(tuned):
    return [[r["order"], r["theta"], r["tile"], r["theta_surface"], round(r["ms"], 4)] +
            [float("%.3g" % r[k]) for k in ("err_p", "worst_p", "err_surface", "worst_surface", "err_force")]
            for r in tuned["table"]]


def swimmer_setting(snaps, steps=5):
    """The mixed-path setting of the swimmer batch and the serving mix: the autotuner over the
    batch's swimmers of grids up to 512^2 (36 of the 64: every phase the small grids hold) and
    the 1024^2 cylinder, errors the largest over them against FP64 references, the surface
    acceptance tuned too."""
    from paper_1610_04398_gb300 import autotune, synth
    reps = autotune.batch_representatives(snaps) + [synth.cylinder_flow(1024, seed=2000)]
    tuned = autotune.autotune(reps, steps=steps)
    b = tuned["best"]
    return {"order": b["order"], "theta": b["theta"], "tile": b["tile"], "theta_surface": b["theta_surface"]}, {
        "best": b, "snapshots": tuned["snapshots"], "reference": tuned["reference"], "tol": tuned["tol"],
        "safety": tuned["safety"], "seconds": round(tuned["seconds"], 2), "table_columns": TUNE_COLUMNS,
        "table": tune_table(tuned)}


def batch_measure(a, flush, snaps, setting, steps=20):
    """The swimmer batch workload: 64 snapshots whose grid side and phase are drawn from
    seed 4000 + k over {256, 512, 1024, 2048}, 4096 surface points each, mixed path at the
    setting tuned on the batch's own swimmers (``swimmer_setting``), every snapshot's step
    graph a branch of one CUDA graph launched once per batch step (pp_batch).  Timed over ``steps`` launches with L2 flushed
    between them, beside the same 64 step graphs launched one after another; errors of every
    snapshot against FP64 references of the same snapshot (grid: the FP64 zero-padded FFT
    solve, the exact discrete sum; surface pressure and forces: the FP64 tree-code at p = 20,
    theta = 0.4)."""
    import torch
    from paper_1610_04398_gb300 import api
    count = len(snaps)
    items = []
    for s in snaps:
        plan = api.Plan(s.n, s.h, setting["order"], setting["theta"], precision="mixed", lift=s.lift, uinf=s.uinf,
                        tile=setting["tile"], theta_surface=setting["theta_surface"])
        f = [torch.from_numpy(np.ascontiguousarray(x)).to("cuda", torch.float32) for x in
             (s.u, s.v, s.chi, s.usx, s.usy)]
        pts = torch.from_numpy(np.ascontiguousarray(s.points)).cuda()
        nrm = torch.from_numpy(np.ascontiguousarray(s.normals)).cuda()
        P = torch.empty(s.n * s.n, dtype=torch.float32, device="cuda")
        per = torch.empty(len(s.points) * 5, dtype=torch.float64, device="cuda")
        F = torch.zeros(6, dtype=torch.float64, device="cuda")
        g = plan.capture_step(*f, s.lam, p_out=P, points=pts, normals=nrm, nu=s.nu, per_point=per, forces=F)
        items.append(dict(snap=s, plan=plan, graph=g, f=f, pts=pts, nrm=nrm, P=P, per=per, F=F))
    batch = api.Batch([it["graph"] for it in items])
    stream = torch.cuda.current_stream()

    def timed(launch):
        for _ in range(3):
            launch()
        torch.cuda.synchronize()
        ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
        torch.cuda._sleep(int(2e8))
        for e0, e1 in ev:
            flush.zero_()
            e0.record(stream)
            launch()
            e1.record(stream)
        torch.cuda.synchronize()
        return sum(e0.elapsed_time(e1) for e0, e1 in ev) / steps

    def one_by_one():
        for it in items:
            it["graph"].launch()

    launches0 = sum(it["plan"].info().launches for it in items)
    ms_batch = timed(batch.launch)
    launches_per_batch = (sum(it["plan"].info().launches for it in items) - launches0) / (steps + 3)
    ms_seq = timed(one_by_one)
    batch.launch()
    torch.cuda.synchronize()
    # errors against FP64 references of the same snapshots
    errs = []
    for it in items:
        s = it["snap"]
        ref = api.Plan(s.n, s.h, 20, 0.4, precision="fp64", lift=s.lift, uinf=s.uinf)
        f64 = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (s.u, s.v, s.chi, s.usx, s.usy)]
        ref.rhs(*f64, s.lam)
        P64 = torch.empty(s.n * s.n, dtype=torch.float64, device="cuda")
        ref.pressure_solve_fft(P64)
        per64 = torch.empty(len(s.points) * 5, dtype=torch.float64, device="cuda")
        F64 = ref.surface_traction(f64[0], f64[1], it["pts"], it["nrm"], s.nu, per_point=per64)
        torch.cuda.synchronize()
        Pg, Pr = it["P"].double(), P64
        ps, pr = it["per"].view(-1, 5)[:, 0], per64.view(-1, 5)[:, 0]
        Fg = it["F"].cpu().numpy()
        fs = max(math.hypot(F64[4], F64[5]), 1e-300)
        errs.append([float(torch.linalg.vector_norm(Pg - Pr) / torch.linalg.vector_norm(Pr)),
                     float((Pg - Pr).abs().max() / Pr.abs().max()),
                     float(torch.linalg.vector_norm(ps - pr) / torch.linalg.vector_norm(pr)),
                     max(abs(Fg[4] - F64[4]), abs(Fg[5] - F64[5])) / fs])
        ref.destroy()
        del f64, P64, per64
    sizes = [it["snap"].n for it in items]
    cells = sum(n * n for n in sizes)
    batch.destroy()
    for it in items:
        it["graph"].destroy()
        it["plan"].destroy()
    e = np.array(errs)
    return {"snapshots": count, "grids": {str(n): sizes.count(n) for n in sorted(set(sizes))},
            "cells": cells, "surface_points": 4096, "setting": setting,
            "ms_per_batch": ms_batch, "solves_per_s": count * 1e3 / ms_batch,
            "cells_per_s": cells * 1e3 / ms_batch, "launches_per_batch": launches_per_batch,
            "one_by_one_ms": ms_seq, "one_by_one_solves_per_s": count * 1e3 / ms_seq,
            "max_err": {"grid_rel_l2": float(e[:, 0].max()), "grid_worst_cell": float(e[:, 1].max()),
                        "surface_rel_l2": float(e[:, 2].max()), "drag_lift": float(e[:, 3].max())},
            "reference": "grid: FP64 zero-padded FFT solve; surface and forces: FP64 tree-code p=20, theta=0.4",
            "l2": "flushed by a 256 MB write before each batch launch",
            "mode": "one CUDA graph launch per batch (each snapshot's step graph a branch)"}


def in_config_measure(a, tuned, snap, dev, pts, nrm, flush):
    """The fastest autotuned setting inside the configuration's own sweep (p in {12, 16, 20},
    theta in {0.4, 0.5, 0.6}) that meets the error bound, timed like the headline: the step
    graph replayed a.steps times, L2 flushed between steps, CUDA events per step."""
    import torch
    from paper_1610_04398_gb300 import api
    rows = [r for r in tuned["table"] if r["ok"] and r["theta"] <= 0.6 and r["order"] in (12, 16, 20)]
    if not rows:
        return None
    best = min(rows, key=lambda r: r["ms"])
    plan = api.Plan(a.n, snap.h, best["order"], best["theta"], precision="mixed", lift=snap.lift,
                    uinf=snap.uinf, tile=best["tile"], theta_surface=best["theta_surface"])
    P = torch.empty(a.n * a.n, dtype=plan.dtype, device="cuda")
    F = torch.zeros(6, dtype=torch.float64, device="cuda")
    g = plan.capture_step(*dev, snap.lam, p_out=P, points=pts, normals=nrm, nu=snap.nu, forces=F)
    for _ in range(max(a.warmup, 3)):
        g.launch()
    torch.cuda.synchronize()
    stream = torch.cuda.current_stream()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(a.steps)]
    torch.cuda._sleep(int(min(2e9, 1.2e5 * a.steps)))
    for e0, e1 in ev:
        flush.zero_()
        e0.record(stream)
        g.launch()
        e1.record(stream)
    torch.cuda.synchronize()
    ms = sum(e0.elapsed_time(e1) for e0, e1 in ev) / a.steps
    g.destroy()
    plan.destroy()
    return {"order": best["order"], "theta": best["theta"], "tile": best["tile"],
            "theta_surface": best["theta_surface"], "ms_per_step": ms,
            "solves_per_s": 1e3 / ms, "err_p_vs_fp64_reference": best["err_p"],
            "err_force_vs_fp64_reference": best["err_force"],
            "note": "fastest setting within theta <= 0.6 meeting the bound, timed like the headline"}


def e2e(a, plan, snap, host, world):
    """The same metric through the C ABI with HOST buffers (pp_pipeline): every step
    copies the five input fields and the surface points host->device from pinned
    memory, solves, and copies the pressure field and the forces back; the copies of
    neighbouring steps overlap the solve (two device slots, three streams).  Timed on
    the host clock from the first submit until the last result is in host memory."""
    import torch
    import torch.distributed as dist
    from paper_1610_04398_gb300 import api
    pinned = [x.pin_memory() for x in host]
    P_host = torch.empty(a.n * a.n, dtype=plan.dtype).pin_memory()
    F_host = torch.empty(6, dtype=torch.float64).pin_memory()
    pts_h = torch.from_numpy(np.ascontiguousarray(snap.points)).pin_memory()
    nrm_h = torch.from_numpy(np.ascontiguousarray(snap.normals)).pin_memory()
    pipe = api.Pipeline(plan, snap.lam, npts=pts_h.shape[0], nu=snap.nu)
    for _ in range(3):
        pipe.submit(*pinned, pts_h, nrm_h, P_host, F_host)
    pipe.wait()
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    t0 = time.perf_counter()
    for _ in range(a.steps):
        pipe.submit(*pinned, pts_h, nrm_h, P_host, F_host)
    pipe.wait()
    t = time.perf_counter() - t0
    pipe.destroy()
    if world > 1:
        tt = torch.tensor([t], device="cuda", dtype=torch.float64)
        dist.all_reduce(tt, op=dist.ReduceOp.MAX)
        t = float(tt.item())
    esz = 4 if a.precision == "mixed" else 8
    return {"value": a.steps * world / t, "unit": "solves/s",
            "h2d_bytes_per_step": 5 * esz * a.n * a.n + 2 * 16 * a.npts,
            "d2h_bytes_per_step": esz * a.n * a.n + 48,
            "mode": "pp_pipeline: pinned host buffers, uploads and downloads overlapping the solve"}


def penal_measure(a, plan, dev, snap, F, peaks):
    """Penalisation force (Eq. dragPenal) on the resident snapshot: the reduction's time
    over 200 calls (CUDA events on the plan's stream, device output), its bytes (the five
    fields) against the HBM peak, and the drag it gives beside the surface-force drag of
    the solve.  L2 is flushed before each call by READING a 256 MB buffer: a write flush
    leaves up to the whole L2 dirty, and a 40 us kernel would mostly time the write-back."""
    import torch
    res = torch.zeros(4, dtype=torch.float64, device="cuda")
    flush = torch.ones(L2_FLUSH_BYTES // 4, dtype=torch.float32, device="cuda")
    sink = torch.empty((), dtype=torch.float32, device="cuda")
    for _ in range(3):
        plan.penal_force(*dev, snap.lam, forces=res)
    torch.cuda.synchronize()
    stream = torch.cuda.current_stream()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(200)]
    torch.cuda._sleep(int(2e8))  # the host queues all calls ahead of the GPU (no launch gaps timed)
    for e0, e1 in ev:
        sink.copy_(flush.sum())
        e0.record(stream)
        plan.penal_force(*dev, snap.lam, forces=res)
        e1.record(stream)
    torch.cuda.synchronize()
    ms = [e0.elapsed_time(e1) for e0, e1 in ev]
    t = statistics.median(ms) / 1e3
    nbytes = 5 * a.n * a.n * (4 if a.precision == "mixed" else 8)
    gbs = nbytes / t / 1e9
    r = res.cpu().numpy()
    return {"ms": t * 1e3, "bytes": nbytes, "achieved_gbs": gbs, "frac_of_hbm": gbs / peaks["hbm_gbs"],
            "drag_penal": float(r[2]), "lift_penal": float(r[3]),
            "drag_surface": float(F[4].item()), "lift_surface": float(F[5].item()),
            "l2": "flushed by a 256 MB read before each call",
            "note": "the synthetic snapshot is not a Navier-Stokes state, so the two drags need not agree"}


def fft_measure(a, plan, peaks, calls=100):
    """Zero-padded FFT (Hockney) solve of the same discrete sum on the whole grid, beside the
    multipole grid solve, both from the source the last step left resident (pp_rhs is not
    part of either): median time over ``calls`` calls each (CUDA events, L2 flushed by a
    256 MB read before each call), the FFT's three-pass HBM bytes and nominal flop count
    (5 N log2 N per complex transform of N points) against the peaks, and the whole-grid
    difference between the two solves."""
    import torch
    nn = a.n * a.n
    M = 2 * a.n
    Pf = torch.empty(nn, dtype=plan.dtype, device="cuda")
    Pm = torch.empty(nn, dtype=plan.dtype, device="cuda")
    plan.pressure_solve_fft(Pf)  # the first call forms the kernel spectrum
    plan.pressure_solve(Pm)
    torch.cuda.synchronize()
    diff = float(torch.linalg.vector_norm((Pm - Pf).double()) / torch.linalg.vector_norm(Pf.double()))
    flush = torch.ones(L2_FLUSH_BYTES // 4, dtype=torch.float32, device="cuda")
    sink = torch.empty((), dtype=torch.float32, device="cuda")
    stream = torch.cuda.current_stream()

    def timed(fn, out):
        for _ in range(3):
            fn(out)
        torch.cuda.synchronize()
        ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(calls)]
        torch.cuda._sleep(int(2e8))
        for e0, e1 in ev:
            sink.copy_(flush.sum())
            e0.record(stream)
            fn(out)
            e1.record(stream)
        torch.cuda.synchronize()
        return statistics.median([e0.elapsed_time(e1) for e0, e1 in ev]) / 1e3

    t_fft = timed(plan.pressure_solve_fft, Pf)
    t_fmm = timed(plan.pressure_solve, Pm)
    esz = 4 if a.precision == "mixed" else 8
    half = (M // 2 + 1) * M * esz                  # transformed kernel, read once
    work = a.n * (a.n + 4) * 2 * esz               # half spectra, written and read twice each
    nbytes = 2 * nn * esz + 4 * work + half
    flops = (a.n + M + 2) * 5.0 * M * math.log2(M)
    gbs = nbytes / t_fft / 1e9
    tf = flops / t_fft / 1e12
    fp32_peak, _ = alu_peak("mixed", torch.cuda.get_device_properties(0).multi_processor_count)
    traffic = recorded_traffic("k_fft_solve", workload_config(a)["workload"])
    return {"ms": t_fft * 1e3, "fmm_grid_solve_ms": t_fmm * 1e3, "fft_over_fmm_speed": t_fmm / t_fft,
            "launches": 3, "bytes_3pass": nbytes, "traffic": traffic,
            "achieved_gbs": gbs, "frac_of_hbm": gbs / peaks["hbm_gbs"],
            "nominal_flops": flops, "achieved_tflops": tf,
            "frac_of_fp32": tf / fp32_peak if a.precision == "mixed" else None,
            "fmm_vs_fft_rel_l2": diff,
            "l2": "flushed by a 256 MB read before each call",
            "note": "both solves start from the same resident source; the FMM time includes its near field"}


def adaptive_work(lv, ix, iy, theta, p):
    """Algorithmic FP64 work of one adaptive solve, from the tree's lists: near-field cell pairs
    between leaves of one level (one multiply-add each, the log comes from the table), between
    leaves of different levels (a multiply-add plus a square root and a log, counted as 2 flop
    here and reported apart), multipole-to-local pairs (the direct form: about 12 p flop for
    each of the p + 1 output terms), and the leaf expansions and local evaluations (8 p flop per
    cell each)."""
    from paper_1610_04398_gb300 import api
    t = api.adaptive_tree(lv, ix, iy, theta)
    leaf_level = np.empty(len(lv), np.int64)
    leaf_level[t["leaf"][t["leaf"] >= 0]] = t["level"][t["leaf"] >= 0]
    same = leaf_level[t["p2p"][:, 0]] == leaf_level[t["p2p"][:, 1]]
    pairs_same, pairs_mixed = int(same.sum()) * 4096, int((~same).sum()) * 4096
    m2l = int(len(t["m2l"]))
    cells = int(len(lv)) * 64
    flop = 2.0 * (pairs_same + pairs_mixed) + 12.0 * p * (p + 1) * m2l + 2 * 8.0 * p * cells
    return {"near_cell_pairs_same_level": pairs_same, "near_cell_pairs_mixed_level": pairs_mixed,
            "m2l_pairs": m2l, "flop": flop}


def adaptive_measure(calls=20):
    """FP64 pressure on an adaptive grid refined towards a cylinder (blocks of 8 x 8 cells,
    levels 3..8: the finest cells 1/2048 of the domain near the body), pp_atree_solve at
    p = 20, theta = 0.5 on a kept tree: median device time per solve (CUDA events), the first
    solve's wall time (tree upload and allocation included) and the tree build, and the
    difference from a solve of the same tree at p = 30 (parity with the oracle's direct sum is
    in tests/test_gpu_adaptive.py)."""
    import torch
    from paper_1610_04398_gb300 import api, synth
    lv, ix, iy = synth.adaptive_blocks(3, 8, centre=(0.3, 0.5), radius=0.05, band=2.0)
    xs, ys, hs = synth.block_cells(lv, ix, iy, cells=8)
    q = (np.random.default_rng(2000).normal(size=xs.size) + 0.5) * hs ** 2
    qd = torch.from_numpy(q).cuda()
    t0 = time.perf_counter()
    tree = api.AdaptiveTree(lv, ix, iy, 0.5)
    t_build = time.perf_counter() - t0
    try:
        t0 = time.perf_counter()
        P = tree.solve(qd, 20)
        torch.cuda.synchronize()
        t_first = time.perf_counter() - t0
        stream = torch.cuda.current_stream()
        ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(calls)]
        for e0, e1 in ev:
            e0.record(stream)
            tree.solve(qd, 20, p_out=P)
            e1.record(stream)
        torch.cuda.synchronize()
        t = statistics.median([e0.elapsed_time(e1) for e0, e1 in ev]) / 1e3
        P30 = tree.solve(qd, 30)
        # the mixed-precision solve of the same tree at p = 12 and p = 20, timed the same way
        qf = qd.float()
        mixed = {}
        for order in (12, 20):
            Pm = tree.solve_mixed(qf, order)
            evm = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(calls)]
            for e0, e1 in evm:
                e0.record(stream)
                tree.solve_mixed(qf, order, p_out=Pm)
                e1.record(stream)
            torch.cuda.synchronize()
            tm = statistics.median([e0.elapsed_time(e1) for e0, e1 in evm]) / 1e3
            err = float(torch.linalg.vector_norm(Pm.double() - P30) / torch.linalg.vector_norm(P30))
            mixed[f"p{order}"] = {"ms": tm * 1e3, "cells_per_s": xs.size / tm, "rel_l2_vs_fp64_p30": err}
        torch.cuda.synchronize()
    finally:
        tree.destroy()
    diff30 = float(torch.linalg.vector_norm(P - P30) / torch.linalg.vector_norm(P30))
    work = adaptive_work(lv, ix, iy, 0.5, 20)
    tflops = work["flop"] / t / 1e12
    pk64, src64 = alu_peak("fp64", 0)
    pkfix, srcfix = fixed_peak(152)
    return {"leaves": int(lv.size), "cells": int(xs.size), "levels": [int(lv.min()), int(lv.max())],
            "ms": t * 1e3, "cells_per_s": xs.size / t, "first_solve_ms": t_first * 1e3,
            "tree_build_ms": t_build * 1e3, "work": work,
            "roofline": {"bound": "alu", "achieved": tflops, "peak": pkfix, "unit": "TFLOP/s",
                         "frac": tflops / pkfix, "peak_source": srcfix, "fp64_peak": pk64, "fp64_peak_source": src64},
            "rel_l2_vs_p30": diff30,
            "mixed": mixed,
            "note": "FP64, p = 20, theta = 0.5; ms: device time of a solve on a kept tree (CUDA events); "
                    "first_solve_ms includes uploading the tree and allocating the expansions; mixed: "
                    "pp_atree_solve_mixed on the same tree (FP32 q and output)"}


# ------------------------------------------------------------------------ serving
def serve_pool(sizes, seed, npts_range=(512, 8192)):
    """Device-resident snapshots for the serving load: every size as a cylinder and as a
    swimmer, surface points drawn uniformly from npts_range (seeded)."""
    import torch
    from paper_1610_04398_gb300 import synth
    synth.set_device("cuda")
    rng = np.random.default_rng(seed)
    pool = []
    for n in sizes:
        for kind in ("cylinder", "swimmer"):
            npts = int(rng.integers(npts_range[0], npts_range[1] + 1))
            if kind == "cylinder":
                snap = synth.cylinder_flow(n, seed=int(rng.integers(1 << 30)), n_surface=npts)
            else:
                snap = synth.swimmer_snapshot(n, float(rng.uniform()), seed=int(rng.integers(1 << 30)),
                                              n_surface=2 * (npts // 2))
            pool.append(snap)
    synth.set_device(None)
    return pool


def serve_run(pool, precision, rate, n_requests, seed, slots=8, budget=150 << 30, order=12, theta=0.6,
              tile=16, theta_surface=0.0, ring=16):
    """Poisson arrivals at ``rate`` req/s (inf: all at once) of random pool snapshots through
    pp_server; returns latency percentiles and throughput from the server's own clock."""
    import torch
    from paper_1610_04398_gb300 import api
    dt = torch.float32 if precision == "mixed" else torch.float64
    dev = []
    for snap in pool:
        f = [torch.from_numpy(np.ascontiguousarray(x)).to("cuda", dt) for x in
             (snap.u, snap.v, snap.chi, snap.usx, snap.usy)]
        pts = torch.from_numpy(np.ascontiguousarray(snap.points)).cuda()
        nrm = torch.from_numpy(np.ascontiguousarray(snap.normals)).cuda()
        outs = [(torch.empty(snap.n * snap.n, dtype=dt, device="cuda"),
                 torch.empty(6, dtype=torch.float64, device="cuda")) for _ in range(ring)]
        dev.append((snap, f, pts, nrm, outs))
    torch.cuda.synchronize()
    srv = api.Server(budget_bytes=budget, slots=slots, precision=precision, order=order, theta=theta, tile=tile,
                     theta_surface=theta_surface)
    rng = np.random.default_rng(seed)
    pick = rng.integers(0, len(pool), n_requests)
    gaps = rng.exponential(1.0 / rate, n_requests) if math.isfinite(rate) else np.zeros(n_requests)
    use = [0] * len(pool)
    ids = []
    # warm the plan cache: every pool entry `slots` times at once, so that the trees a
    # saturated mix needs are resident before timing
    warm = []
    for k, (snap, f, pts, nrm, outs) in enumerate(dev):
        for j in range(slots):
            warm.append(srv.submit(snap.n, snap.h, *f, snap.lam, nu=snap.nu, lift=snap.lift, uinf=snap.uinf,
                                   points=pts, normals=nrm, p_out=outs[j % ring][0], forces=outs[j % ring][1]))
    for rid in warm:
        srv.wait(rid, 600.0)
    t_next = time.perf_counter()
    for k in range(n_requests):
        t_next += gaps[k]
        while True:
            d = t_next - time.perf_counter()
            if d <= 0:
                break
            time.sleep(min(d, 0.0005) if d > 0.001 else 0)
        e = int(pick[k])
        snap, f, pts, nrm, outs = dev[e]
        P, F = outs[use[e] % ring]
        use[e] += 1
        ids.append(srv.submit(snap.n, snap.h, *f, snap.lam, nu=snap.nu, lift=snap.lift, uinf=snap.uinf,
                              points=pts, normals=nrm, p_out=P, forces=F))
    for rid in ids:
        srv.wait(rid, 600.0)
    times = np.array([srv.query(rid)[2] for rid in ids])
    stats = srv.stats()
    srv.destroy()
    lat = (times[:, 2] - times[:, 0]) * 1e3
    span = times[:, 2].max() - times[:, 0].min()
    return {"rate": rate if math.isfinite(rate) else "saturated", "requests": n_requests,
            "p50_ms": float(np.percentile(lat, 50)), "p99_ms": float(np.percentile(lat, 99)),
            "solves_per_s": n_requests / span, "failed": stats["failed"],
            "plans_resident": stats["plans_resident"], "bytes_held": stats["bytes_held"]}


SERVE_RATES = (50.0, 100.0, 200.0, 500.0, 1000.0, 2000.0)


def serve_summary(a, requests=2000, setting=None):
    """The serving workload: a pool of cylinder and swimmer snapshots on grids of
    256^2-4096^2 (one of each kind per size, surface points drawn from U[512, 8192]);
    ``requests`` Poisson-arrival requests per rate, rates 50-2000 req/s, plans admitted
    against a 150 GB budget, mixed path at ``setting`` (the one tuned on swimmers, which
    meets the bound on both kinds; the headline's when absent); plus the saturated
    throughput of the mixed path and of the plain FP64 path (p = 20, theta = 0.5)."""
    t0 = time.perf_counter()
    pool = serve_pool((256, 512, 1024, 2048, 4096), seed=5001)
    t_pool = time.perf_counter() - t0
    kw = dict(setting) if setting else dict(order=a.order, theta=a.theta, tile=a.tile, theta_surface=a.theta_surface)
    runs = {f"poisson_{int(r)}": serve_run(pool, "mixed", r, requests, seed=int(r), **kw) for r in SERVE_RATES}
    sat = serve_run(pool, "mixed", float("inf"), requests, seed=2, **kw)
    fp64 = serve_run(pool, "fp64", float("inf"), 200, seed=3, order=20, theta=0.5)
    return {"pool": "cylinder+swimmer at 256,512,1024,2048,4096 (npts U[512,8192])", "budget_gb": 150,
            "requests_per_rate": requests, "mixed_setting": kw, **runs,
            "saturated_mixed": sat, "saturated_fp64_p20": fp64,
            "mixed_over_fp64_solves": sat["solves_per_s"] / fp64["solves_per_s"],
            "pool_s": t_pool, "wall_s": time.perf_counter() - t0}


def serve_sweep(a):
    """The serving workload alone (``--serve-sweep``), as one JSON line."""
    import torch
    torch.cuda.set_device(0)
    out = {"metric": "serve latency p50/p99 and solves/s", "unit": "ms / solves/s",
           "serve": serve_summary(a)}
    print(json.dumps(out), flush=True)


# ------------------------------------------------------------------- oracle (CPU)
def oracle_sample_seconds(a, snap, k_targets, seed, k_surf=None):
    """Oracle on a bounded sample of one solve: the full RHS, the exact FP64 sum at
    k_targets random cells and at every surface point (or at k_surf random ones), the
    tractions.  Returns the extrapolated seconds of one whole solve (n^2 + npts targets)
    and the sample time."""
    import oracle
    t0 = time.perf_counter()
    f = oracle.rhs(snap.u, snap.v, snap.chi, snap.usx, snap.usy, h=snap.h, lam=snap.lam)
    q = oracle.source_weights(f, snap.h)
    t_rhs = time.perf_counter() - t0
    rng = np.random.default_rng(seed)
    cells = rng.choice(a.n * a.n, size=k_targets, replace=False)
    c = (np.arange(a.n) + 0.5) * snap.h
    xt, yt = c[cells % a.n], c[cells // a.n]
    t0 = time.perf_counter()
    oracle.green_sum_grid(q, snap.h, xt, yt)
    t_cells = time.perf_counter() - t0
    npts = len(snap.points)
    sel = np.arange(npts) if k_surf is None or k_surf >= npts else rng.choice(npts, size=k_surf, replace=False)
    t0 = time.perf_counter()
    Pk = oracle.green_sum_grid(q, snap.h, snap.points[sel, 0], snap.points[sel, 1])
    t_psurf = time.perf_counter() - t0
    Ps = np.zeros(npts)
    Ps[sel] = Pk
    t0 = time.perf_counter()
    oracle.traction(snap.u, snap.v, snap.h, snap.points, snap.normals, Ps, snap.nu, lift=snap.lift,
                    uinf=snap.uinf)
    t_trac = time.perf_counter() - t0
    per_target = t_cells / k_targets
    total = t_rhs + per_target * a.n * a.n + t_psurf * npts / len(sel) + t_trac
    return total, t_rhs + t_cells + t_psurf + t_trac


def oracle_pairs_per_s_1thread(snap, k_targets=32, seed=7):
    """The oracle's Green's sum on one host thread: exact FP64 sums at k_targets random cells
    over all n^2 sources (pairs per second)."""
    import oracle
    f = oracle.rhs(snap.u, snap.v, snap.chi, snap.usx, snap.usy, h=snap.h, lam=snap.lam)
    q = oracle.source_weights(f, snap.h)
    n = snap.n
    cells = np.random.default_rng(seed).choice(n * n, size=k_targets, replace=False)
    c = (np.arange(n) + 0.5) * snap.h
    t0 = time.perf_counter()
    oracle.green_sum_grid(q, snap.h, c[cells % n], c[cells // n], nthreads=1)
    return k_targets * n * n / (time.perf_counter() - t0)


def cpu_baseline(a, snap):
    import oracle
    oracle.build()
    cores = oracle.max_threads()
    k = a.cpu_targets
    total, sample_s = oracle_sample_seconds(a, snap, k, 99)
    one = oracle_pairs_per_s_1thread(snap)
    return {"value": 1.0 / total, "unit": "solves/s", "cores": cores, "kind": "oracle",
            "sample": (f"full RHS + exact FP64 Green's sum at {k} random cells of {a.n}^2 and at all "
                       f"{a.npts} surface points + tractions ({sample_s:.1f} s); whole-solve time "
                       f"extrapolated by target count ({total:.0f} s per solve)"),
            "pairs_per_s": (k + a.npts) * a.n * a.n / max(sample_s, 1e-9),
            "pairs_per_s_1thread": one}


def run_reference(a):
    rank, world, _ = dist_env()
    if rank != 0:
        return
    import oracle
    from paper_1610_04398_gb300 import synth
    oracle.build()
    cores = oracle.max_threads()
    snap = synth.cylinder_flow(a.n, seed=2000, n_surface=a.npts)
    k, ks = 256, 64
    for i in range(a.warmup):
        oracle_sample_seconds(a, snap, 32, i, k_surf=8)
    per = []
    t0 = time.perf_counter()
    for i in range(a.steps):
        total, _ = oracle_sample_seconds(a, snap, k, 1000 + i, k_surf=ks)
        per.append(total)
    wall = time.perf_counter() - t0
    value = a.steps / sum(per)
    out = {"metric": METRIC, "value": value, "unit": "solves/s", "n_gpus": world, "steps": a.steps,
           "warmup": a.warmup, "ms_per_step": 1e3 * sum(per) / a.steps, "higher_is_better": True,
           "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
           "config": dict(workload_config(a), order=None, theta=None, tile=None,
                          method="exact FP64 direct sum (the oracle)"), "impl": "reference",
           "cpu_baseline": {"value": value, "unit": "solves/s", "cores": cores, "kind": "oracle",
                            "sample": (f"each step: full RHS + exact FP64 sum at {k} random cells and "
                                       f"{ks} of the {a.npts} surface points + tractions; solve time "
                                       f"extrapolated by target count; wall {wall:.1f} s")},
           "e2e": {"value": value, "unit": "solves/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(out), flush=True)


def main():
    a = parse()
    if a.steps is None:
        a.steps = 10 if a.impl == "reference" else 2000
    if a.warmup is None:
        a.warmup = 3 if a.impl == "reference" else 20
    if a.serve_sweep:
        serve_sweep(a)
        return
    if a.impl == "reference":
        run_reference(a)
    else:
        run_ours(a)


if __name__ == "__main__":
    main()
