#!/usr/bin/env python3
"""Throughput of the scenario-batched Split Bellman update on GB300.

Workload (one step = one pass of the whole Split path over one batch):
  giant tour n=500, coords uniform fp32 in [0,100)^2 (depot (50,50)), Q=200,
  S=10^6 demand scenarios per GPU, demands iid U{1..30} int32 (seed 1),
  through sdp_split_eval: tour prep -> pipelined DP kernel (producer warps
  permute demand tiles into tour order in an L2-resident slot ring, DP warps
  run the deque step; + plain fallback, a no-op here) writing fp32 costs and
  uint16 predecessors -> FP64 mean.
Metric: Bellman arc relaxations/s (capacity-feasible arcs (p,i) of Eq. eqdpA,
  counted exactly on the device once, outside the timed region) and
  scenarios/s, whole job over all ranks.
  Inputs (2.0 GB per GPU) are larger than L2 (129 MB): no flush is needed.

  python bench.py [--gpus N --steps K --warmup W] [--impl reference]

N>1 (torchrun, one process per GPU): rank r evaluates scenarios
[r*S, (r+1)*S) of one N*S-scenario set (weak scaling); the global FP64 mean
is the one exchange step (an all-reduce of the per-rank sum).
--impl reference times the FP64 CPU oracle (the paper's method as plain C)
on bounded samples of the same workload on rank 0's host cores.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "Bellman arc relaxations/s (Split, n=500, S=1e6 per GPU)"
UNIT = "arcs/s"
WORKLOAD = "split_n500_Q200_S1e6_U1-30"
BATCH_TOURS = 0  # 0: the full 4096-tour batched workload


def host_cores() -> int:
    try:
        return len(os.sched_getaffinity(0))
    except AttributeError:  # pragma: no cover
        return os.cpu_count() or 1


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            return json.load(f), "measured"
    return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "sm_max_mhz": 2070.0}, "fallback"


class ClockSampler:
    """nvidia-smi clocks / throttle reasons sampled during the timed region."""
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int, interval_ms: int = 20):
        self.gpu = gpu_index
        self.interval_ms = interval_ms
        self.proc = None
        self.lines = []
        self.t = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.gpu}", f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", str(self.interval_ms)],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
            return
        self.t = threading.Thread(target=self._read, daemon=True)
        self.t.start()

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append((time.time(), line.strip()))

    def stop(self):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
        if self.t:
            self.t.join(timeout=2)

    def summary(self, t0, t1):
        rows = []
        for ts, ln in self.lines:
            parts = [x.strip() for x in ln.split(",")]
            if len(parts) < 9:
                continue
            rows.append((ts, parts))
        inside = [r for ts, r in rows if t0 <= ts <= t1] or [r for _, r in rows]
        if not inside:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"],
                    "samples": 0}

        def num(x):
            try:
                return float(x)
            except ValueError:
                return None
        sm = [num(r[1]) for r in inside if num(r[1]) is not None]
        smax = [num(r[2]) for r in inside if num(r[2]) is not None]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[k] for r in inside for k in range(4)
                          if r[5 + k].lower() == "active"})
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(smax) if smax else None, "reasons": reasons,
                "samples": len(inside), "interval_ms": self.interval_ms,
                "window": "timed region" if any(t0 <= ts <= t1 for ts, _ in rows)
                          else "whole sampler run (no sample inside the timed region)"}


# ----------------------------------------------------------------- CPU oracle
def oracle_sample(spec, rows, nthreads):
    """Time the FP64 oracle on demand rows [rows] of the workload."""
    import oracle
    from paper_2602_05179_gb300 import workloads as wl
    tour, xy, _ = wl.split_tour(spec)
    q = wl.split_demands(spec, 0, rows)
    oracle.split(tour, spec.Q, q[:8], coords=xy, nthreads=nthreads)  # build + warm
    t0 = time.perf_counter()
    r = oracle.split(tour, spec.Q, q, coords=xy, want_pred=True, nthreads=nthreads)
    dt = time.perf_counter() - t0
    return int(r["arcs"].sum()), dt


def cpu_baseline(spec, budget_s=12.0):
    import oracle
    cores = min(host_cores(), oracle.max_threads())
    arcs, dt = oracle_sample(spec, 2000, cores)
    rows = int(min(spec.S, max(2000, 2000 * budget_s / max(dt, 1e-3))))
    arcs, dt = oracle_sample(spec, rows, cores)
    return {"value": arcs / dt, "unit": UNIT, "cores": cores, "kind": "oracle",
            "sample": f"first {rows} of the 10^6 scenarios ({arcs} arcs, {dt:.2f} s), "
                      f"FP64 C oracle, OpenMP over scenarios",
            "scenarios_per_s": rows / dt}


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    import oracle
    from paper_2602_05179_gb300 import workloads as wl
    spec = wl.SPLIT_C2
    cores = min(host_cores(), oracle.max_threads())
    # per-step sample sized so the whole run stays within ~90 s
    _, dt = oracle_sample(spec, 512, cores)
    per_scen = dt / 512
    rows = int(max(32, min(20000, 90.0 / max(1, args.steps + args.warmup) / per_scen)))
    tour, xy, _ = wl.split_tour(spec)
    total_arcs, total_t = 0, 0.0
    for k in range(args.warmup + args.steps):
        s0 = (k * rows) % (spec.S - rows)
        q = wl.split_demands(spec, s0, s0 + rows)
        t0 = time.perf_counter()
        r = oracle.split(tour, spec.Q, q, coords=xy, want_pred=True, nthreads=cores)
        dt = time.perf_counter() - t0
        if k >= args.warmup:
            total_arcs += int(r["arcs"].sum())
            total_t += dt
    value = total_arcs / total_t
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT,
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * total_t / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOAD, "n": spec.n, "Q": spec.Q,
                       "scenarios_per_step": rows, "sample": "bounded"},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
                             "sample": f"{rows} scenarios per step, {args.steps} steps"},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line))
    return 0


# ------------------------------------------------------------ oracle checks
# Per-result errors of the GPU results against the FP64 oracle on a seeded
# sample of each workload, taken outside every timed region.  Like the
# cpu_baseline leg they run the oracle on the host (--no-cpu-baseline skips
# both).  Predecessors and policies are compared where the oracle's optimum
# is unique by more than MARGIN relative; costs and values are relative
# errors (the tolerance is 1e-5).
MARGIN = 1e-4


def _rel(c, oc):
    fin = np.isfinite(oc) & np.isfinite(c)
    rel = np.abs(c[fin] - oc[fin]) / np.maximum(np.abs(oc[fin]), 1e-300)
    out = {"sample": int(len(oc)),
           "max_rel_err": float(rel.max()) if rel.size else 0.0,
           "mean_rel_err": float(rel.mean()) if rel.size else 0.0,
           "infeasible_differ": int((np.isinf(c) != np.isinf(oc)).sum())}
    if rel.size:
        m, om = float(c[fin].mean()), float(oc[fin].mean())
        out["rel_err_of_mean"] = abs(m - om) / max(abs(om), 1e-300)
    return out


def split_errors(cost, pred, orc):
    """cost fp32 [k] and pred int64 [k, n] (or None) of the sampled scenarios;
    orc = oracle.split(..., want_margin=True) on the same rows."""
    out = _rel(np.asarray(cost, np.float64), orc["cost"])
    if pred is not None:
        op = orc["pred"].astype(np.int64)
        mask = (op >= 0) & (orc["margin"] > MARGIN)
        out["pred_checked"] = int(mask.sum())
        out["pred_mismatch"] = int((np.asarray(pred)[mask] != op[mask]).sum())
    return out


def reinsert_errors(value, policy, orc, cons, U, I0):
    """value fp32 [k], policy uint8 [k, T] of the sampled scenarios; orc =
    oracle.reinsert(..., want_margin=True) (or reinsert_routes).  Policies are
    compared along the oracle's optimal path at days whose decision is unique
    by more than MARGIN; after a near-tie where the two differ the paths part
    and the comparison of that scenario stops."""
    out = _rel(np.asarray(value, np.float64), orc["value"])
    op, mg = orc["policy"], orc["margin"]
    checked = mism = 0
    for s in range(op.shape[0]):
        I = I0
        for t in range(op.shape[1]):
            if mg[s, t, I] > MARGIN:
                checked += 1
                mism += int(policy[s, t] != op[s, t])
            elif policy[s, t] != op[s, t]:
                break
            I = max(0, (U if op[s, t] else I) - int(cons[s, t]))
    out["policy_checked"] = checked
    out["policy_mismatch"] = mism
    return out


def sample_rows(S, k, seed):
    return np.sort(np.random.default_rng(seed).choice(S, min(k, S), replace=False))


# ----------------------------------------------------------------- GPU arm
def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=2000)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--algo", default="pipe", choices=["pipe", "deque", "stream", "plain"])
    ap.add_argument("--plain-steps", type=int, default=10)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--e2e-steps", type=int, default=20)
    ap.add_argument("--only", default="",
                    choices=["", "reinsert", "routes", "batch", "adjoint", "soft", "fleet", "saa"],
                    help="run one operator line alone (profiling)")
    ap.add_argument("--preds", default="u16", choices=["u16", "i32", "none"])
    ap.add_argument("--no-operators", action="store_true",
                    help="skip the reinsertion / batched / adjoint operator lines")
    ap.add_argument("--batch-tours", type=int, default=0,
                    help="override the batched line's tour count (its first B tours; small "
                         "cases for ncu captures)")
    ap.add_argument("--scenarios", type=int, default=0,
                    help="override S per GPU (small cases for ncu captures)")
    args = ap.parse_args()
    global BATCH_TOURS
    BATCH_TOURS = args.batch_tours
    if args.warmup < 3:
        ap.error("--warmup must be >= 3")
    if args.impl == "reference":
        return run_reference(args)

    import torch
    import torch.distributed as dist

    from paper_2602_05179_gb300 import api
    from paper_2602_05179_gb300 import workloads as wl

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if args.only:
        print(json.dumps(operators(api, wl, dev, only=args.only, steps=args.steps,
                                   checks=not args.no_cpu_baseline)))
        return 0
    if world > 1:
        dist.init_process_group("nccl", device_id=dev)

    spec = wl.SPLIT_C2
    if args.scenarios > 0:
        import dataclasses
        spec = dataclasses.replace(spec, S=args.scenarios)
    S = spec.S
    tour, xy, _ = wl.split_tour(spec)
    t_d = torch.from_numpy(tour).to(dev)
    c_d = torch.from_numpy(xy).to(dev)
    from paper_2602_05179_gb300 import shard
    s0, s1 = shard.scenario_range(rank, world, S)
    q_d = wl.split_demands_device(spec, dev, s0, s1)
    _, total = api.split_count_arcs(t_d, spec.Q, q_d, coords=c_d, per_scenario=False)
    torch.cuda.synchronize()
    arcs_rank = int(total)

    preds = None if args.preds == "none" else args.preds

    def step(algo=args.algo):
        return api.split_eval(t_d, spec.Q, q_d, coords=c_d, preds=preds, algo=algo)

    # ---- device-resident timed region
    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    ks = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    ke = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    for ev in ks + ke:  # create the CUDA events before the timed region
        ev.record()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    clocks = ClockSampler(local)
    clocks.start()
    time.sleep(0.3)
    torch.cuda.synchronize()
    t_wall0 = time.time()
    e0.record()
    for k in range(args.steps):
        api.set_profile_events(ks[k], ke[k])
        r = step()
    e1.record()
    torch.cuda.synchronize()
    t_wall1 = time.time()
    if world > 1:
        dist.barrier()
    clocks.stop()
    ms_total = e0.elapsed_time(e1)
    kern_ms = statistics.mean(a.elapsed_time(b) for a, b in zip(ks, ke))
    flags = api.status()
    t = torch.tensor([ms_total, kern_ms], dtype=torch.float64, device=dev)
    cnt = torch.tensor([float(arcs_rank), float(r["cost"].double().sum())],
                       dtype=torch.float64, device=dev)
    if world > 1:
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        dist.all_reduce(cnt, op=dist.ReduceOp.SUM)
    ms_total, kern_ms = float(t[0]), float(t[1])
    arcs_all = cnt[0].item()
    ms_step = ms_total / args.steps
    value = arcs_all * args.steps / (ms_total / 1e3)
    scen_s = S * world * args.steps / (ms_total / 1e3)

    # ---- plain-kernel comparison (same call, algo=plain)
    plain = None
    if args.plain_steps > 0:
        for _ in range(3):
            step("plain")
        torch.cuda.synchronize()
        p0 = torch.cuda.Event(enable_timing=True)
        p1 = torch.cuda.Event(enable_timing=True)
        p0.record()
        for _ in range(args.plain_steps):
            step("plain")
        p1.record()
        torch.cuda.synchronize()
        pms = p0.elapsed_time(p1) / args.plain_steps
        plain = {"value": arcs_rank * world / (pms / 1e3), "unit": UNIT, "ms_per_step": pms,
                 "speedup_over_plain": (pms / ms_step)}

    # ---- end to end through the public API with host buffers
    e2e = None
    if args.e2e_steps > 0:
        e2e = e2e_run(args, api, spec, t_d, c_d, q_d, arcs_all, world, dist, dev)

    if rank != 0:
        if world > 1:
            dist.destroy_process_group()
        return 0
    errors = None
    if not args.no_cpu_baseline:
        errors = headline_errors(spec, tour, xy, r, s0, s1)
    ops = None
    if not args.no_operators and world == 1:
        del q_d, r
        torch.cuda.empty_cache()
        ops = operators(api, wl, dev, checks=not args.no_cpu_baseline)
    return report(args, spec, S, world, value, scen_s, ms_step, kern_ms, arcs_all, plain,
                  e2e, flags, clocks, t_wall0, t_wall1, dist, ops, errors)


def _preds_i64(p):
    a = p.cpu().numpy()
    if a.dtype == np.int16:  # uint16 bits; 0xFFFF is the infeasible sentinel
        a = a.astype(np.int64) & 0xFFFF
        a[a == 0xFFFF] = -1
    return a.astype(np.int64)


def headline_errors(spec, tour, xy, r, s0, s1):
    """The last timed step's costs and predecessors on 2,000 sampled
    scenarios of this rank against the FP64 oracle."""
    import torch
    import oracle
    from paper_2602_05179_gb300 import workloads as wl
    rows = sample_rows(s1 - s0, 2000, 11)
    q = np.concatenate([wl.split_demands(spec, s0 + int(k), s0 + int(k) + 1) for k in rows])
    orc = oracle.split(tour, spec.Q, q, coords=xy, want_margin=True)
    idx = torch.from_numpy(rows).to(r["cost"].device)
    pred = _preds_i64(r["pred"][idx]) if r.get("pred") is not None else None
    return split_errors(r["cost"][idx].cpu().numpy(), pred, orc)


def e2e_run(args, api, spec, t_d, c_d, q_d, arcs_all, world, dist, dev):
    import torch
    q_host = torch.empty(q_d.shape, dtype=torch.int32, pin_memory=True)
    q_host.copy_(q_d)
    h2d = q_host.numel() * 4
    preds = None if args.preds == "none" else args.preds
    # the public call with host demands: the library copies them chunk by
    # chunk behind the evaluation; the per-scenario costs and the mean come
    # back to pinned host buffers (the predecessors stay on the device)
    cost_host = torch.empty(q_d.shape[0], dtype=torch.float32, pin_memory=True)
    mean_host = torch.empty((), dtype=torch.float64, pin_memory=True)

    def once():
        r = api.split_eval(t_d, spec.Q, q_host, coords=c_d, preds=preds, algo=args.algo)
        cost_host.copy_(r["cost"], non_blocking=True)
        mean_host.copy_(r["mean"], non_blocking=True)
        torch.cuda.current_stream().synchronize()
        return float(mean_host)
    for _ in range(3):
        once()
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    w0 = time.perf_counter()
    for _ in range(args.e2e_steps):
        once()
    w1 = time.perf_counter()
    et = torch.tensor([w1 - w0], dtype=torch.float64, device=dev)
    if world > 1:
        dist.all_reduce(et, op=dist.ReduceOp.MAX)
    return {"value": arcs_all * args.e2e_steps / float(et[0]), "unit": UNIT,
            "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": cost_host.numel() * 4 + 8,
            "steps": args.e2e_steps, "copies": "demands in (pinned host memory, chunked by "
            "the library); costs and mean out (pinned host buffers)"}


def _timed(fn, steps, warmup=3, events=True):
    """(ms per call, mean kernel ms via the profile hook) on the current stream."""
    import torch
    from paper_2602_05179_gb300 import api
    for _ in range(warmup):
        fn()
    torch.cuda.synchronize()
    ks = [torch.cuda.Event(enable_timing=True) for _ in range(steps)]
    ke = [torch.cuda.Event(enable_timing=True) for _ in range(steps)]
    for ev in ks + ke:
        ev.record()
    a = torch.cuda.Event(enable_timing=True)
    b = torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    a.record()
    for k in range(steps):
        if events:
            api.set_profile_events(ks[k], ke[k])
        fn()
    b.record()
    torch.cuda.synchronize()
    kern = statistics.mean(x.elapsed_time(y) for x, y in zip(ks, ke)) if events else None
    return a.elapsed_time(b) / steps, kern


class OpCtx:
    """What every operator line needs: the binding, the workloads, the device,
    the step count, whether to run the oracle checks, and the peaks."""

    def __init__(self, api, wl, dev, steps, checks):
        import torch
        self.api, self.wl, self.dev, self.steps, self.checks = api, wl, dev, steps, checks
        peaks, self.peak_src = measured_peaks()
        self.sms = torch.cuda.get_device_properties(dev).multi_processor_count
        self.p_alu = self.sms * 128 * peaks.get("sm_max_mhz", 2070.0) * 1e6
        self.hbm = peaks["hbm_gbs"]

    def alu_roof(self, ops, kms):
        a = ops / (kms / 1e3)
        return {"bound": "alu", "achieved": a, "peak": self.p_alu, "unit": "ops/s",
                "frac": a / self.p_alu,
                "peak_source": f"{self.sms} SMs x 128 lanes x sm_max_mhz ({self.peak_src})"}

    def hbm_roof(self, byts, kms):
        a = byts / (kms / 1e3) / 1e9
        return {"bound": "hbm", "achieved": a, "peak": self.hbm, "unit": "GB/s",
                "frac": a / self.hbm, "peak_source": f"{self.peak_src} hbm_gbs (copy)"}


def operators(api, wl, dev, only="", steps=0, checks=True):
    """The other hot-path operators at their workload sizes (few steps each),
    each with its plain-kernel comparison and, with checks, its errors
    against the oracle on a sample."""
    import torch
    c = OpCtx(api, wl, dev, steps, checks)
    fns = {"reinsert": op_reinsert, "routes": op_routes, "adjoint": op_adjoint,
           "soft": op_soft, "fleet": op_fleet, "batch": op_batch, "saa": op_saa}
    out = {}
    for k in ([only] if only else list(fns)):
        fns[k](c, out)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
    return out


def op_reinsert(c, out):
    """Reinsertion T=60, U=200, S=10^6: the default kernel (the reachable
    states, one scenario per lane) against the one-scenario-per-warp kernel,
    which evaluates every state."""
    import torch
    rs = c.wl.REINSERT_C3
    cons = c.wl.reinsert_consumption_device(rs, c.dev)
    fixed_h = c.wl.reinsert_fixed(rs)
    fixed = torch.from_numpy(fixed_h).to(c.dev)

    def run(algo):
        return c.api.reinsert_eval(rs.T, rs.U, rs.I0, rs.h, rs.p, rs.unit_cost, fixed, cons,
                                   algo=algo)
    ms, kms = _timed(lambda: run("auto"), c.steps or 10)
    r = run("auto")
    wms, wkms = _timed(lambda: run("warp"), 5)
    rw = run("warp")
    line = {"value": rs.S / (ms / 1e3), "unit": "scenarios/s", "ms_per_step": ms, "kernel_ms": kms,
            "kernel": "reinsert_chain_kernel (reachable states, one scenario per lane)",
            # credits the at most t + 1 states that day t can start in
            "roofline": c.alu_roof(2 * rs.S * sum(min(t + 1, rs.U + 1) for t in range(rs.T)), kms),
            "vs_plain": {"kernel": "reinsert_kernel (one scenario per warp)",
                         "ms_per_step": wms, "kernel_ms": wkms, "speedup": wkms / kms,
                         "values_bit_identical": bool(torch.equal(r["value"], rw["value"])),
                         "policies_bit_identical": bool(torch.equal(r["policy"], rw["policy"]))}}
    if c.checks:
        import oracle
        rows = sample_rows(rs.S, 2000, 12)
        ch = np.concatenate([c.wl.reinsert_consumption(rs, int(k), int(k) + 1) for k in rows])
        orc = oracle.reinsert(rs.T, rs.U, rs.I0, rs.h, rs.p, rs.unit_cost, fixed_h, ch,
                              want_margin=True)
        idx = torch.from_numpy(rows).to(c.dev)
        line["errors"] = reinsert_errors(r["value"][idx].cpu().numpy(),
                                         r["policy"][idx].cpu().numpy(), orc, ch, rs.U, rs.I0)
    out[rs.name] = line


def op_routes(c, out):
    """Reinsertion with K = 4 route options per day."""
    import torch
    rr = c.wl.REINSERT_ROUTES
    cons = c.wl.reinsert_consumption_device(rr, c.dev)
    cap = c.wl.reinsert_route_caps_device(rr, c.dev)
    rcost_h = c.wl.reinsert_route_costs(rr)
    rcost = torch.from_numpy(rcost_h).to(c.dev)
    K = int(rcost.shape[1])

    def run(algo="auto"):
        return c.api.reinsert_eval(rr.T, rr.U, rr.I0, rr.h, rr.p, rr.unit_cost, None, cons,
                                   route_cost=rcost, route_cap=cap, algo=algo)
    ms, kms = _timed(run, c.steps or 10)
    r = run()
    wms, wkms = _timed(lambda: run("warp"), c.steps or 10)
    rw = run("warp")
    same = all(bool(torch.equal(r[k], rw[k])) for k in ("value", "policy"))
    line = {"value": rr.S / (ms / 1e3), "unit": "scenarios/s", "ms_per_step": ms, "kernel_ms": kms,
            "kernel": "reinsert_chain_kernel (route options, reachable states, one scenario per lane)",
            "roofline": c.alu_roof(2 * rr.S * (K + 1) * sum(min(t + 1, rr.U + 1) for t in range(rr.T)), kms),
            "vs_warp": {"kernel": "reinsert_routes_kernel (one scenario per warp)", "ms_per_step": wms,
                        "kernel_ms": wkms, "speedup": wkms / kms, "bit_identical": same}}
    if c.checks:
        import oracle
        rows = sample_rows(rr.S, 500, 13)
        ch = np.concatenate([c.wl.reinsert_consumption(rr, int(k), int(k) + 1) for k in rows])
        caph = np.concatenate([c.wl.reinsert_route_caps(rr, int(k), int(k) + 1) for k in rows])
        orc = oracle.reinsert_routes(rr.T, rr.U, rr.I0, rr.h, rr.p, rr.unit_cost, rcost_h,
                                     caph, ch, want_margin=True)
        idx = torch.from_numpy(rows).to(c.dev)
        line["errors"] = reinsert_errors(r["value"][idx].cpu().numpy(),
                                         r["policy"][idx].cpu().numpy(), orc, ch, rr.U, rr.I0)
    out[rr.name] = line


def op_adjoint(c, out):
    """Split adjoint n=300, S=10^5: the fused forward + on-chip backtrack,
    one step = a CUDA graph replay of the whole adjoint (the kernel's own
    time from an eager call through the profile hook), against the plain
    kernel's forward with stored predecessors + their backtrack."""
    import torch
    ad = c.wl.ADJOINT_C5
    tour, xy, distm = c.wl.split_tour(ad)
    t = torch.from_numpy(tour).to(c.dev)
    dm = torch.from_numpy(distm).to(c.dev)
    q = c.wl.split_demands_device(ad, c.dev)
    _, tot = c.api.split_count_arcs(t, ad.Q, q, dist=dm, per_scenario=False)
    arcs = int(tot)
    g1 = torch.ones((), dtype=torch.float32, device=c.dev)
    fn = lambda: c.api.split_backward(t, ad.Q, q, dm, g1, want_hist=True)
    eager_ms, kms = _timed(fn, c.steps or 20)
    graphed = c.api.GraphedSplitBackward(t, ad.Q, q, dm, g1, want_hist=True)
    ms, _ = _timed(graphed.run, c.steps or 20, events=False)
    g, hist = fn()
    torch.cuda.synchronize()
    graph_same = bool(torch.equal(graphed.grad, g) and torch.equal(graphed.hist, hist))
    byts = ad.S * ad.n * 4

    def plain():
        p = c.api.split_eval(t, ad.Q, q, dist=dm, algo="plain", preds="i32")["pred"]
        return c.api.split_backward(t, ad.Q, q, dm, g1, pred=p, pred_dtype="i32",
                                    want_hist=True)
    pms, _ = _timed(plain, 3, events=False)
    gp, hp = plain()
    line = {"value": arcs / (ms / 1e3), "unit": "arcs/s (forward+backtrack)",
            "ms_per_step": ms, "kernel_ms": kms, "kernel": "split_tmem_adj_kernel",
            "launch": "CUDA graph replay of the step (hist reset, tour prep, DP kernel, "
                      "recompute of flagged scenarios, gradient assembly)",
            "eager_ms_per_step": eager_ms, "graph_bits_equal_eager": graph_same,
            "roofline": c.hbm_roof(byts, kms),
            "alu_frac": 2 * arcs / (kms / 1e3) / c.p_alu,
            "vs_plain": {"path": "plain forward with int32 predecessors + backtrack kernel",
                         "ms_per_step": pms, "speedup": pms / ms,
                         "route_counts_equal": bool(torch.equal(hist, hp)),
                         "grad_max_abs_diff": float((g - gp).abs().max())}}
    if c.checks:
        import oracle
        qh = c.wl.split_demands(ad)
        orc = oracle.split(tour, ad.Q, qh, dist=distm)
        go = oracle.split_mean_grad(tour, orc["pred"])
        start, end, _ = oracle.split_route_counts(orc["pred"])
        h = hist.cpu().numpy()
        gd = g.cpu().double().numpy()
        line["errors"] = {"sample": ad.S,
                          "grad_max_abs_err": float(np.abs(gd - go).max()),
                          "route_count_abs_diff": int(np.abs(h[:ad.n] - start).sum() +
                                                      np.abs(h[ad.n:] - end).sum()),
                          "note": "against the oracle's own optimal splits of all 10^5 "
                                  "scenarios; counts differ only at near-ties"}
    out[ad.name] = line


def op_soft(c, out):
    """Soft-capacity Split: the bench workload (n=500, Q=200, S=10^6,
    U{1..30}) with 10 per unit of route load above Q; the pipelined kernel
    (AUTO: hard window in the deque, expired entries as one running minimum),
    beside the DEQUE soft kernel (the same recursion and bits) and PLAIN
    (every pair (p, i) relaxed), the latter on the first 65,536 scenarios."""
    import torch
    spec = c.wl.SPLIT_C2
    beta = 10.0
    tour, xy, _ = c.wl.split_tour(spec)
    t = torch.from_numpy(tour).to(c.dev)
    cc = torch.from_numpy(xy).to(c.dev)
    q = c.wl.split_demands_device(spec, c.dev)
    fn = lambda: c.api.split_eval(t, spec.Q, q, coords=cc, preds="u16", algo="pipe",
                                  overload_penalty=beta)
    ms, kms = _timed(fn, c.steps or 20)
    r = fn()
    fnd = lambda: c.api.split_eval(t, spec.Q, q, coords=cc, preds="u16", algo="deque",
                                   overload_penalty=beta)
    dms, dkms = _timed(fnd, c.steps or 20)
    rd = fnd()
    same = bool(torch.equal(r["cost"], rd["cost"]) and torch.equal(r["pred"], rd["pred"]))
    n, S = spec.n, spec.S
    byts = S * n * 4 + S * 4 + S * n * 2
    sub = 65536
    qs = q[:sub]
    fnp = lambda: c.api.split_eval(t, spec.Q, qs, coords=cc, preds="u16", algo="plain",
                                   overload_penalty=beta)
    pms, _ = _timed(fnp, 2, warmup=1, events=False)
    line = {"value": S / (ms / 1e3), "unit": "scenarios/s", "ms_per_step": ms,
            "kernel_ms": kms, "kernel": "split_pipe_kernel (soft)",
            "roofline": c.hbm_roof(byts, kms),
            "vs_deque": {"kernel": "split_tmem_soft_kernel", "ms_per_step": dms, "kernel_ms": dkms,
                         "speedup": dkms / kms, "bit_identical": same},
            "vs_plain": {"plain_ms_per_65536": pms, "plain_scenarios_per_s": sub / (pms / 1e3),
                         "speedup": (S / (ms / 1e3)) / (sub / (pms / 1e3))}}
    if c.checks:
        import oracle
        rows = sample_rows(S, 1000, 14)
        qh = np.concatenate([c.wl.split_demands(spec, int(k), int(k) + 1) for k in rows])
        orc = oracle.split_soft(tour, spec.Q, beta, qh, coords=xy, want_margin=True)
        idx = torch.from_numpy(rows).to(c.dev)
        line["errors"] = split_errors(r["cost"][idx].cpu().numpy(), _preds_i64(r["pred"][idx]),
                                      orc)
    out["split_soft_n500_S1e6_beta10"] = line


def band_states(q, tour, Q, K):
    """States (k, i) of each scenario from which a split into at most K routes
    can still finish: i lies between what k routes reach from the start and
    what K - k reach back from the end (0 where no such split exists)."""
    n = len(tour)
    out = np.zeros(len(q), np.int64)
    for s, row in enumerate(np.asarray(q, np.int64)[:, np.asarray(tour) - 1]):
        if (row > Q).any():
            continue
        L = np.concatenate([[0], np.cumsum(row)])
        hi, lo = [0], [n]
        for _ in range(K):
            hi.append(int(np.searchsorted(L, L[hi[-1]] + Q, side="right")) - 1)
            lo.append(int(np.searchsorted(L, L[lo[-1]] - Q, side="left")))
        if lo[K] == 0:
            out[s] = sum(max(0, hi[k] - max(lo[K - k], 1) + 1) for k in range(1, K + 1))
    return out


def op_fleet(c, out):
    """Fleet-limited Split (at most K = 42 routes) on the Split benchmark's
    recipe (n = 500, Q = 200, U{1..30}) with S = 65,536: the limit binds
    (about 39-42 routes are needed).  The kernel evaluates the band of states
    that K routes leave, counted here on 256 scenarios; the plain comparison
    runs every feasible p of every layer, one thread per scenario, on 4,096
    scenarios."""
    import dataclasses
    import torch
    K, S = 42, 65536
    spec = dataclasses.replace(c.wl.SPLIT_C2, S=S)
    tour, xy, _ = c.wl.split_tour(spec)
    t = torch.from_numpy(tour).to(c.dev)
    cc = torch.from_numpy(xy).to(c.dev)
    q = c.wl.split_demands_device(spec, c.dev, 0, S)
    fn = lambda: c.api.split_fleet_eval(t, spec.Q, q, K, coords=cc)
    ms, kms = _timed(fn, c.steps or 5)
    c.api.status()
    r = fn()
    fell_back = bool(c.api.status() & c.api.FLAG_FALLBACK)
    Sp = 4096
    qp = q[:Sp].contiguous()
    pms, pkms = _timed(lambda: c.api.split_fleet_eval(t, spec.Q, qp, K, coords=cc, algo="plain"),
                       1, warmup=1)
    rp = c.api.split_fleet_eval(t, spec.Q, qp, K, coords=cc, algo="plain")
    torch.cuda.synchronize()
    same = all(bool(torch.equal(r[k][:Sp], rp[k])) for k in ("cost", "nroutes", "route"))
    fin = torch.isfinite(r["cost"])
    states = band_states(q[:: S // 256].cpu().numpy(), tour, spec.Q, K).mean()
    line = {"value": S / (ms / 1e3), "unit": "scenarios/s", "ms_per_step": ms, "kernel_ms": kms,
            "kernel": "split_fleet_band_kernel (one warp per scenario, positions across lanes)",
            "max_routes": K, "feasible_frac": float(fin.float().mean()),
            "flagged_recomputed": fell_back,
            "recompute": "scenarios with windows of more than 32 positions: the same kernel in wider "
                         "blocks, inside ms_per_step",
            # demands in; cost, route count and each customer's route out
            "roofline": c.hbm_roof(S * (spec.n * 4 + 4 + 4 + spec.n), kms),
            "band_states_per_scenario": float(states), "states_per_s": float(states) * S / (kms / 1e3),
            "vs_plain": {"path": "one thread per scenario, every feasible p of every layer",
                         "sample": Sp, "kernel_ms": pkms,
                         "speedup_per_scenario": (pkms / Sp) / (kms / S),
                         "bit_identical": same}}
    if c.checks:
        import oracle
        rows = sample_rows(S, 128, 21)
        qh = np.concatenate([c.wl.split_demands(spec, int(k), int(k) + 1) for k in rows])
        orc = oracle.split_fleet(tour, spec.Q, K, qh, coords=xy, want_margin=True)
        idx = torch.from_numpy(rows).to(c.dev)
        line["errors"] = _rel(r["cost"][idx].cpu().numpy().astype(np.float64), orc["cost"])
        uniq = np.isfinite(orc["cost"]) & (orc["margin"] > 1e-5)
        nr = r["nroutes"][idx].cpu().numpy()
        ro = r["route"][idx].cpu().numpy().astype(np.int64)
        line["errors"]["routes_checked"] = int(uniq.sum())
        line["errors"]["route_mismatch"] = int((ro[uniq] != orc["route"][uniq]).any(1).sum() +
                                               (nr[uniq] != orc["nroutes"][uniq]).sum())
    out[f"fleet_n500_Q200_K{K}_S65536"] = line


def op_batch(c, out):
    """Batched Split: 4096 tours, n ~ U{20..1000}, S=4096 (persistent launch,
    CUDA graph, autotuned), against the plain kernel run once per tour."""
    import tempfile
    import torch
    bs = c.wl.BATCH_C4
    if BATCH_TOURS and BATCH_TOURS != bs.B:
        import dataclasses
        bs = dataclasses.replace(bs, B=BATCH_TOURS, name=f"batch_B{BATCH_TOURS}_n20-1000_S4096")
    nb = c.wl.batch_sizes(bs)
    tours, coords = zip(*(c.wl.batch_tour(bs, b, int(nb[b])) for b in range(bs.B)))
    dem_off = np.zeros(bs.B, np.int64)
    dem_off[1:] = np.cumsum(nb[:-1].astype(np.int64) * bs.S)
    total = int(dem_off[-1] + nb[-1] * bs.S)
    d = torch.empty(total, dtype=torch.int32, device=c.dev)
    for b in range(bs.B):
        seg = d[dem_off[b]:dem_off[b] + nb[b] * bs.S].view(bs.S, int(nb[b]))
        c.wl.batch_demands_device(bs, b, int(nb[b]), seg)
    tt = torch.from_numpy(np.concatenate(tours)).to(c.dev)
    cc = torch.from_numpy(np.concatenate(coords)).to(c.dev)
    plan = c.api.SplitPlan(nb, tt, cc, d, bs.Q, bs.S, dem_off=dem_off)
    arcs = plan.count_arcs()
    tune = plan.autotune(os.path.join(tempfile.gettempdir(), "sdp_autotune_cache.txt"))
    ms, _ = _timed(plan.run, c.steps or 10, events=False)
    kms = plan.kernel_ms()
    costs, _ = plan.run()
    costs = costs.clone()
    byts = total * 4 + bs.B * bs.S * 4
    line = {"value": arcs / (ms / 1e3), "unit": UNIT,
            "scenarios_per_s": bs.B * bs.S / (ms / 1e3), "ms_per_step": ms,
            "kernel_ms_last_replay": kms, "arcs_per_step": arcs, "launch": tune,
            "roofline": c.hbm_roof(byts, kms), "alu_frac": 2 * arcs / (kms / 1e3) / c.p_alu}
    # the plain kernel once per tour (4096 launches), same inputs
    toff = np.concatenate([[0], np.cumsum(nb[:-1].astype(np.int64))])
    coff = np.concatenate([[0], np.cumsum(nb[:-1].astype(np.int64) + 1)])
    pc = torch.empty_like(costs)

    def per_tour():
        for b in range(bs.B):
            n = int(nb[b])
            r = c.api.split_eval(tt[toff[b]:toff[b] + n], bs.Q,
                                 d[dem_off[b]:dem_off[b] + n * bs.S].view(bs.S, n),
                                 coords=cc[coff[b]:coff[b] + n + 1], algo="plain", mean=False)
            pc[b].copy_(r["cost"])
    pms, _ = _timed(per_tour, 1, warmup=1, events=False)
    relp = ((costs.double() - pc.double()).abs() / pc.double().abs().clamp_min(1e-30))
    line["vs_plain"] = {"path": "plain kernel, one launch per tour", "ms_per_step": pms,
                        "speedup": pms / ms, "max_rel_diff": float(relp.max()),
                        "over_1e-5": int((relp > 1e-5).sum())}
    if c.checks:
        import oracle
        rng = np.random.default_rng(15)
        sel = rng.choice(bs.B, min(16, bs.B), replace=False)
        errs = []
        for b in sel:
            n = int(nb[b])
            rows = sample_rows(bs.S, 256, 16 + int(b))
            qh = np.concatenate([c.wl.batch_demands(bs, int(b), n, int(k), int(k) + 1)
                                 for k in rows])
            orc = oracle.split(tours[b], bs.Q, qh, coords=coords[b], want_margin=True)
            errs.append((costs[int(b)][torch.from_numpy(rows).to(c.dev)].cpu().numpy(),
                         orc["cost"]))
        cg = np.concatenate([e[0] for e in errs])
        co = np.concatenate([e[1] for e in errs])
        line["errors"] = _rel(cg.astype(np.float64), co)
        line["errors"]["sample"] = f"{len(sel)} tours x 256 scenarios"
    plan.close()
    out[bs.name] = line


def op_saa(c, out):
    """SAA candidate search on one CVRPSD instance (n=100, Q=100, Poisson(10)
    demands, S=10^4): every iteration scores the current tour and 1024
    neighbours in one batched-plan replay and takes the best strict
    improvement on the device.  Arcs are counted per iteration on a replay
    of the same (deterministic) move stream, outside the timed run."""
    import tempfile
    import torch
    spec = c.wl.SAA_C6
    tour, xy, _ = c.wl.split_tour(spec)
    t = torch.from_numpy(tour).to(c.dev)
    cc = torch.from_numpy(xy).to(c.dev)
    q = c.wl.split_demands_device(spec, c.dev)
    cache = os.path.join(tempfile.gettempdir(), "sdp_autotune_cache.txt")
    s = c.api.SaaSearch(t, cc, q, spec.Q, c.wl.SAA_B, seed=spec.seed)
    shape = s.autotune(cache)
    warm = 3
    s.run(warm)  # warm-up: graph capture, first moves
    torch.cuda.synchronize()
    iters = c.steps or 20
    a = torch.cuda.Event(enable_timing=True)
    b = torch.cuda.Event(enable_timing=True)
    a.record()
    trace, acc = s.run(iters)
    b.record()
    torch.cuda.synchronize()
    ms = a.elapsed_time(b)
    final_tour, _ = s.state()
    s.close()
    # the same iterations again, one at a time, counting the arcs scored
    s2 = c.api.SaaSearch(t, cc, q, spec.Q, c.wl.SAA_B, seed=spec.seed)
    s2.autotune(cache)
    s2.run(warm)
    arcs = 0
    for _ in range(iters):
        s2.run(1)
        arcs += s2.count_arcs()
    s2.close()
    evals = iters * (c.wl.SAA_B + 1)
    tr = trace.cpu().numpy()
    line = {"value": iters * c.wl.SAA_B / (ms / 1e3), "unit": "candidates/s",
            "ms_per_iteration": ms / iters, "iterations": iters,
            "scenario_evaluations_per_s": evals * spec.S / (ms / 1e3),
            "arcs_per_s": arcs / (ms / 1e3), "arcs": arcs,
            # the scenarios in, the costs out and in again for the means
            "roofline": c.hbm_roof(iters * (spec.S * spec.n * 4 + (c.wl.SAA_B + 1) * spec.S * 8), ms),
            "best_mean_first": float(tr[0]), "best_mean_last": float(tr[-1]),
            "improving_iterations": int((acc >= 0).sum()),
            "launch": shape}
    line["roofline"]["note"] = ("whole iterations (moves, plan replay, selection) timed; bound by instruction "
                                "issue, and arcs of beginnings that a neighbour shares with the current "
                                "tour are scored without being run")
    if c.checks:
        import oracle
        ft = final_tour.cpu().numpy()
        orc = oracle.split(ft, spec.Q, c.wl.split_demands(spec), coords=xy, want_pred=False)
        line["errors"] = {"sample": spec.S, "best_mean_rel_err":
                          abs(float(tr[-1]) - orc["mean"]) / abs(orc["mean"])}
    out[f"saa_n{spec.n}_S1e4_B{c.wl.SAA_B}"] = line


def issue_roof(tj, S, kern_ms, sms, sm_mhz):
    """The DP kernel against its instruction-issue bound: the warp
    instructions of one launch (the stored capture's smsp__inst_executed.sum,
    scaled from the captured scenario count to S) over the kernel time,
    against SMs x 4 schedulers x the maximum SM clock (one warp instruction
    per scheduler per cycle).  None without a matching capture."""
    inst = (tj or {}).get("smsp_inst_executed_captured")
    cap = (tj or {}).get("captured_scenarios")
    if not inst or not cap or not kern_ms or kern_ms <= 0 or not sms or not sm_mhz:
        return None
    per_launch = float(inst) * float(S) / float(cap)
    peak = float(sms) * 4.0 * float(sm_mhz) * 1e6
    achieved = per_launch / (kern_ms / 1e3)
    return {"bound": "issue", "achieved": achieved, "peak": peak,
            "unit": "warp instructions/s", "frac": achieved / peak,
            "inst_per_launch": per_launch,
            "source": "smsp__inst_executed.sum of the stored capture, scaled by scenarios",
            "peak_source": f"{sms} SMs x 4 schedulers x sm_max_mhz"}


def report(args, spec, S, world, value, scen_s, ms_step, kern_ms, arcs_all, plain, e2e,
           flags, clocks, t_wall0, t_wall1, dist, ops=None, errors=None):
    import torch
    dev = torch.device("cuda", torch.cuda.current_device())
    peaks, peak_src = measured_peaks()
    n = spec.n
    pbytes = {"u16": 2, "i32": 4, "none": 0}[args.preds]
    alg_bytes = S * n * 4 + S * 4 + S * n * pbytes  # demands in, fp32 cost + preds out
    achieved = alg_bytes / (kern_ms / 1e3) / 1e9
    traffic = None
    tj_now = None  # the stored capture, when it describes the kernel being timed
    tp = os.path.join(ROOT, "profiles", "split_pipe_traffic.json" if args.algo == "pipe"
                      else "split_deque_traffic.json")
    if os.path.exists(tp):
        with open(tp) as f:
            tj = json.load(f)
        if tj.get("kernel_rev") == kernel_rev(args.algo):
            traffic = tj.get("dram_bytes_per_launch")
            tj_now = tj
    roof = {"bound": "hbm", "achieved": achieved, "peak": peaks["hbm_gbs"], "unit": "GB/s",
            "frac": achieved / peaks["hbm_gbs"], "traffic": traffic,
            "kernel": {"pipe": "split_pipe_kernel", "deque": "split_tmem_kernel",
                       "plain": "split_plain_kernel",
                       "stream": "stream_prep_kernel + split_stream_kernel"}[args.algo],
            "kernel_ms": kern_ms,
            "algorithmic_bytes_per_launch": alg_bytes, "peak_source": f"{peak_src} hbm_gbs (copy)"}
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    p_alu = sms * 128 * peaks.get("sm_max_mhz", 2070.0) * 1e6
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_step,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32", "data": "synthetic",
        "config": {"workload": WORKLOAD if S == 1_000_000 else f"split_n500_Q200_S{S}_U1-30",
                   "n": n, "Q": spec.Q, "S_per_gpu": S,
                   "demand": "iid U{1..30} int32, seed 1", "coords": "U[0,100)^2 fp32",
                   "algo": args.algo, "preds": args.preds,
                   "parallelism": f"scenario-sharded x{world}",
                   "l2": "inputs larger than L2 (2.0 GB demands per step), no flush",
                   "arcs_per_step": arcs_all},
        "scenarios_per_s": scen_s,
        "roofline": roof,
        "alu_roofline": {"ops_per_arc": 2, "peak_ops_per_s": p_alu,
                         "frac": 2 * arcs_all / world / (kern_ms / 1e3) / p_alu},
        "issue_roofline": issue_roof(tj_now, S, kern_ms, sms, peaks.get("sm_max_mhz", 2070.0)),
        "vs_plain": plain,
        "errors": errors,
        "e2e": e2e,
        "gpu_launches": 5 * args.steps,
        "device_flags": flags,
        "operators": ops,
        "clocks": clocks.summary(t_wall0, t_wall1),
    }
    if not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(spec)
    print(json.dumps(line))
    if world > 1:
        dist.destroy_process_group()
    return 0


def kernel_rev(algo="pipe"):
    """Hash of the DP kernel source's code (comments and blank lines left
    out), to tell whether stored ncu counters still describe the kernel being
    timed."""
    import hashlib
    import re
    name = {"pipe": "split_pipe.cu", "stream": "split_stream.cu"}.get(algo, "split_deque.cu")
    src = os.path.join(ROOT, "paper_2602_05179_gb300", "csrc", name)
    with open(src) as f:
        code = re.sub(r"//[^\n]*", "", f.read())
    code = "\n".join(line.rstrip() for line in code.splitlines() if line.strip())
    return hashlib.sha256(code.encode()).hexdigest()[:16]


if __name__ == "__main__":
    sys.exit(main())
