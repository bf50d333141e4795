#!/usr/bin/env python
"""Benchmark of the GranQ fake-quantization hot path on B200.

One step = fused forward + backward fake-quantization (range -> scale / zero-point ->
quantize / clamp / dequantize -> STE backward, one library call per tensor) of every tensor
of the ResNet-18 and MobileNetV2 ImageNet-shaped activation sets (12 fp32 tensors, batch
128) at both of their bit-widths (4 and 5): 24 calls, 914 M elements, 14.6 GB of
algorithmic traffic (16 B per element: read x, read gy, write y, write gx).  A step runs all
twelve tensors at 4 bits, then all twelve at 5 bits, so no tensor is touched by two
consecutive calls and every call finds its tensor cold (7.3 GB pass through between them).

Prints ONE JSON line.  `value` is algorithmic GB/s over K eagerly launched steps with all
tensors resident in HBM (mean; median and best step beside it); `e2e` is the same metric
through the host-buffer entry point (pinned host memory, copies inside the timed region);
`roofline` relates the dominant kernel to the measured HBM copy bandwidth; `per_tensor` is each
call's sustained cold time (back-to-back calls over rotating copies of the tensor, no event
between them); `sub` holds bounded runs of the other configurations, entry points, group modes
and plans; `cpu_baseline` is the CPU oracle timed on a bounded sample of the same workload.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]
With --gpus N > 1 and no torchrun environment the script starts its N ranks itself.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from paper_2503_18339_b200 import workloads as wl  # noqa: E402

METRIC = "fake-quant fwd+bwd GB/s (algorithmic bytes: 16 B/element fp32)"
UNIT = "GB/s"
WORKLOAD = ("configs 3+4: ResNet-18 + MobileNetV2 ImageNet-shaped activations, batch 128, fp32, "
            "12 tensors x b in {4,5}, fused fwd+bwd, channel groups over (n,h,w)")
BYTES_PER_ELEM = 16
NOMINAL_HBM_GBS = 8000.0
FALLBACK_HBM_GBS = 6650.0
CPU_SAMPLE = "cfg3.1-3.4 ([128,64,56,56] [128,128,28,28] [128,256,14,14] [128,512,7,7]), b=4 and b=5, fused fwd+bwd"


def workload_specs():
    return wl.config_tensors(3) + wl.config_tensors(4)


def measured_peak():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as fh:
            return float(json.load(fh)["hbm_gbs"]), "measured (MEASURED_PEAKS.json hbm_gbs)"
    except Exception:
        return FALLBACK_HBM_GBS, "fallback (6.65 TB/s, earlier measurement on this pool)"


DOMINANT_KERNEL_SOURCES = ("granq_colteam.cu", "granq_device.cuh")


def kernel_source_hash() -> str:
    """Hash of the files the dominant kernel is compiled from."""
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_2503_18339_b200", "csrc")
    for name in DOMINANT_KERNEL_SOURCES:
        with open(os.path.join(csrc, name), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def recorded_traffic():
    """DRAM bytes per launch of the dominant kernel from the committed ncu summary, or None
    when there is none or the kernel sources have changed since it was taken."""
    path = os.path.join(ROOT, "profiles", "colteam_kernel_traffic.txt")
    try:
        with open(path) as fh:
            rec = json.load(fh)
        if rec.get("kernel_source_hash") != kernel_source_hash():
            return None
        return rec
    except Exception:
        return None


class ClockSampler:
    """Samples SM clocks and throttle reasons with nvidia-smi while the timed region runs."""
    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.rows = []
        self.proc = None
        self.thread = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "100"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None
            return
        self.thread = threading.Thread(target=self._read, daemon=True)
        self.thread.start()

    def _read(self):
        for line in self.proc.stdout:
            self.rows.append((time.time(), [c.strip() for c in line.split(",")]))

    def stop(self, t0: float, t1: float):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        time.sleep(0.15)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        rows = [r for (t, r) in self.rows if t0 <= t <= t1 + 0.2 and len(r) >= 7] or \
               [r for (_, r) in self.rows if len(r) >= 7]
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        sm = [float(r[0]) for r in rows]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = [n for i, n in enumerate(names) if any(r[3 + i].lower().startswith("active") for r in rows)]
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": float(rows[0][1]), "reasons": reasons,
                "samples": len(rows), "power_w_max": max(float(r[2]) for r in rows)}


def max_over_ranks(ms: float, device: str = "cuda") -> float:
    """The slowest rank's device time (every rank gets it); the identity when not distributed."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return float(ms)
    t = torch.tensor([ms], device=device, dtype=torch.float64)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_gbs(bytes_per_step_per_rank: int, world: int, ms_per_step: float) -> float:
    """Aggregate algorithmic GB/s of `world` replicas that each process one step in ms_per_step."""
    return world * bytes_per_step_per_rank / (ms_per_step * 1e-3) / 1e9


def time_oracle(specs_bits, arrays=None):
    """Seconds the CPU oracle needs for fused fwd+bwd on the given (spec, bits) list; elements processed.
    `arrays` maps spec.name -> (x, gy) numpy arrays already generated."""
    from oracle import granq_oracle as orc
    orc.lib()
    elems, secs = 0, 0.0
    cache = dict(arrays or {})
    for spec, bits in specs_bits:
        if spec.name not in cache:
            cache[spec.name] = (wl.make_activation(spec), wl.make_upstream_grad(spec))
        x, gy = cache[spec.name]
        t = time.perf_counter()
        orc.fused(x, bits, gy=gy, want_codes=False)
        secs += time.perf_counter() - t
        elems += spec.numel
    return secs, elems


def cpu_sample():
    specs = wl.config_tensors(3)[1:]
    return [(s, b) for s in specs for b in s.bits]


def run_reference(args):
    """The CPU oracle as the reference arm: each step is the bounded sample of the workload."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    sample = cpu_sample()
    for _ in range(min(args.warmup, 1)):
        time_oracle(sample[:1])
    total_s, total_e = 0.0, 0
    for _ in range(args.steps):
        s, e = time_oracle(sample)
        total_s += s
        total_e += e
    value = total_e * BYTES_PER_ELEM / total_s / 1e9
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * total_s / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": WORKLOAD, "step": "bounded sample: " + CPU_SAMPLE},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle", "sample": CPU_SAMPLE},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        "elements_per_s": total_e / total_s,
    }
    print(json.dumps(line))


def free_port() -> int:
    import socket
    with socket.socket() as sk:
        sk.bind(("127.0.0.1", 0))
        return sk.getsockname()[1]


def spawn_ranks(n: int, argv, extra_env=None, timeout=None):
    """Start `n` ranks of `argv` on this node (RANK / LOCAL_RANK / WORLD_SIZE / MASTER_* set as torchrun
    would) and wait for them; returns their exit codes.  Rank 0 inherits stdout."""
    port = free_port()
    procs = []
    for r in range(n):
        env = dict(os.environ, RANK=str(r), LOCAL_RANK=str(r), WORLD_SIZE=str(n), MASTER_ADDR="127.0.0.1",
                   MASTER_PORT=str(port), **(extra_env or {}))
        procs.append(subprocess.Popen(list(argv), env=env, stdout=None if r == 0 else subprocess.DEVNULL))
    codes = []
    for pr in procs:
        try:
            codes.append(pr.wait(timeout=timeout))
        except subprocess.TimeoutExpired:
            pr.kill()
            codes.append(-9)
    return codes


def rank_selftest():
    """The multi-rank plumbing without a GPU: gloo ranks agree on the slowest rank's time and rank 0 prints
    the aggregate (what the spawn path of --gpus N is tested with on CPU)."""
    import torch.distributed as dist
    rank, world = int(os.environ["RANK"]), int(os.environ["WORLD_SIZE"])
    dist.init_process_group("gloo", rank=rank, world_size=world)
    ms = max_over_ranks(10.0 * (rank + 1), device="cpu")
    if rank == 0:
        print(json.dumps({"selftest": True, "n_gpus": world, "ms_per_step": ms,
                          "value": whole_job_gbs(1_000_000_000, world, ms)}))
    dist.barrier()
    dist.destroy_process_group()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--e2e-steps", type=int, default=2)
    ap.add_argument("--e2e-lanes", type=int, default=2, help="streams (each with its own arena) the end-to-end "
                                                             "calls rotate over")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-sub", action="store_true", help="skip the bounded sub-records and the per-tensor pass")
    ap.add_argument("--table", action="store_true", help="also print a per-tensor table to stderr")
    ap.add_argument("--tune", default="", help="planner overrides for experiments, e.g. depth=3,max_buf_units=4000")
    ap.add_argument("--plan", default="auto", choices=["auto", "two_pass", "naive", "staged", "l2wave", "colwalk",
                                                       "cluster"],
                    help="force an execution plan of the fused entry point (experiments)")
    ap.add_argument("--op", default="fused", choices=["fused", "range", "fwd", "bwd", "fused_fwd_packmask",
                                                      "bwd_packmask"],
                    help="time another entry point instead of the fused one (bytes/element 4, 8, 12; 8.125 for the "
                         "two halves of the mask-carrying split)")
    ap.add_argument("--no-graph", action="store_true", help="skip the CUDA-graph replay figure")
    ap.add_argument("--clear-workspace", action="store_true",
                    help="let every call clear its workspace (one more memset node per call) instead of "
                         "passing GRANQ_FLAG_WORKSPACE_ZEROED")
    ap.add_argument("--sharded", action="store_true", help="also time the batch-sharded forward / backward "
                                                           "(range, all-reduce of the range, forward with packed "
                                                           "mask, backward from the mask)")
    ap.add_argument("--only", default="", help="profiling aid: keep only workload tensors whose name contains this")
    ap.add_argument("--rank-selftest", action="store_true", help=argparse.SUPPRESS)
    args = ap.parse_args()
    if args.rank_selftest:
        if "RANK" not in os.environ:
            codes = spawn_ranks(args.gpus, [sys.executable, os.path.abspath(__file__)] + sys.argv[1:])
            sys.exit(max(abs(c) for c in codes))
        rank_selftest()
        return
    if args.impl == "reference":
        if args.steps > 3:
            args.steps = 3          # each step is ~10 s of CPU work
        run_reference(args)
        return
    if args.gpus > 1 and "WORLD_SIZE" not in os.environ:
        # a plain `python bench.py --gpus N`: start the N ranks here (one per GPU, NCCL for the barrier and the
        # maximum over ranks only: the path has no exchange step)
        codes = spawn_ranks(args.gpus, [sys.executable, os.path.abspath(__file__)] + sys.argv[1:])
        sys.exit(max(abs(c) for c in codes))

    import torch
    import torch.distributed as dist
    from paper_2503_18339_b200 import binding as b

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    b.lib()
    knob_ids = {"depth": b.KNOB_STAGED_DEPTH, "max_buf_units": b.KNOB_STAGED_MAX_BUF_UNITS,
                "grid": b.KNOB_STAGED_GRID, "ctas_per_sm": b.KNOB_STAGED_CTAS_PER_SM,
                "l2_wave_kb": b.KNOB_L2_WAVE_KB, "l2_upl": b.KNOB_L2_UPL, "l2_ctas_per_sm": b.KNOB_L2_CTAS_PER_SM,
                "l2_lag": b.KNOB_L2_LAG, "cl_tile_kb": b.KNOB_CLUSTER_TILE_KB, "cl_ctas": b.KNOB_CLUSTER_CTAS,
                "cl_threads": b.KNOB_CLUSTER_THREADS, "cl_load": b.KNOB_CLUSTER_LOAD,
                "cl_prefetch": b.KNOB_CLUSTER_PREFETCH, "cl_kmul": b.KNOB_CLUSTER_KMUL,
                "cl_early_launch": b.KNOB_CLUSTER_EARLY_LAUNCH, "col_team": b.KNOB_COLWALK_TEAM}
    for item in filter(None, args.tune.split(",")):
        name, val = item.split("=")
        b.tune(knob_ids[name], int(val))
    warmup = max(args.warmup, 3)
    plan_flags = {"auto": 0, "two_pass": b.FLAG_FORCE_TWO_PASS, "naive": b.FLAG_FORCE_NAIVE,
                  "staged": b.FLAG_FORCE_STAGED, "l2wave": b.FLAG_FORCE_L2WAVE,
                  "colwalk": b.FLAG_FORCE_COLWALK, "cluster": b.FLAG_FORCE_CLUSTER}[args.plan]
    flags = plan_flags
    if not args.clear_workspace:      # the workspaces are cleared once below and every call leaves them clear
        flags |= b.FLAG_WORKSPACE_ZEROED
    peak, peak_src = measured_peak()

    specs = [s for s in workload_specs() if args.only in s.name]
    # ---- host (pinned) inputs and outputs; every rank has its own batch (weak scaling, no exchange) ----
    host = []
    for s in specs:
        xs = torch.empty(s.shape, dtype=torch.float32).pin_memory()
        gs = torch.empty(s.shape, dtype=torch.float32).pin_memory()
        wl.make_activation(s, out=xs.numpy(), block_offset=1000 * rank)
        wl.make_upstream_grad(s, out=gs.numpy(), block_offset=1000 * rank)
        host.append((xs, gs))

    def outputs_for(x, groups, group=b.GROUP_CHANNEL):
        return b.FakeQuantOut(y=torch.empty_like(x), gx=torch.empty_like(x),
                              lo=torch.empty(groups, device="cuda"), hi=torch.empty(groups, device="cuda"),
                              workspace=b.make_workspace(x, group=group, zeroed=True))

    dev = []
    for s, (xs, gs) in zip(specs, host):
        x = xs.cuda(non_blocking=True)
        gy = gs.cuda(non_blocking=True)
        dev.append((x, gy, outputs_for(x, s.shape[1])))
    torch.cuda.synchronize()
    # all tensors at their first bit-width, then all at their second: consecutive calls never share a tensor
    nbits = max(len(s.bits) for s in specs)
    calls = [(i, s.bits[k]) for k in range(nbits) for i, s in enumerate(specs) if k < len(s.bits)]
    elems_per_step = sum(specs[i].numel for i, _ in calls)
    plans = [b.fused_plan(b.F32, specs[i].shape, flags=plan_flags) for i, _ in calls]
    launches_per_step = sum(n for _, n in plans)
    stream = torch.cuda.Stream()          # a stream of its own: the legacy default stream cannot be captured
    torch.cuda.set_stream(stream)

    bpe = {"fused": 16, "range": 4, "fwd": 8, "bwd": 12, "fused_fwd_packmask": 8.125, "bwd_packmask": 8.125}[args.op]
    bytes_per_step = int(elems_per_step * bpe)
    if args.op.endswith("packmask"):
        for x, gy, out in dev:
            out.packed_mask = b.make_packed_mask(x)
    if args.op != "fused":          # the stand-alone entry points need a range: take each tensor's own
        for x, gy, out in dev:
            b.granq_fakequant_fused(x, 4, gy=gy, out=out, stream=stream)
            if args.op == "bwd_packmask":
                b.granq_fakequant_fused_fwd_packmask(x, 4, out=out, stream=stream)

    def one_call(x, gy, out, bits, op=None, fl=None, group=b.GROUP_CHANNEL):
        op = args.op if op is None else op
        fl = flags if fl is None else fl
        if op == "fused":
            b.granq_fakequant_fused(x, bits, gy=gy, group=group, out=out, flags=fl, stream=stream)
        elif op == "fused_fwd":
            b.granq_fakequant_fused(x, bits, group=group, out=out, flags=fl, stream=stream)
        elif op == "range":
            b.granq_range(x, lo=out.lo, hi=out.hi, workspace=out.workspace, stream=stream)
        elif op == "fwd":
            b.granq_fakequant_fwd(x, bits, out.lo, out.hi, y=out.y, stream=stream)
        elif op == "fused_fwd_packmask":
            b.granq_fakequant_fused_fwd_packmask(x, bits, out=out, flags=fl, stream=stream)
        elif op == "bwd_packmask":
            b.granq_fakequant_bwd_packmask(gy, out.packed_mask, gx=out.gx, stream=stream)
        else:
            b.granq_fakequant_bwd(gy, x, bits, out.lo, out.hi, gx=out.gx, stream=stream)

    def step(events=None):
        for ci, (i, bits) in enumerate(calls):
            x, gy, out = dev[i]
            if events is not None:
                events[ci].record(stream)
            one_call(x, gy, out, bits)
        if events is not None:
            events[len(calls)].record(stream)

    def check_status():
        torch.cuda.synchronize()
        for _, _, out in dev:
            assert b.workspace_status(out.workspace) == b.OK

    for _ in range(warmup):
        step()
    check_status()

    def barrier():
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()

    # ---- timed region: K eagerly launched steps, device time, max over ranks ----
    # One event per step boundary gives the per-step times (median, best).  The first steps also carry one event
    # before every call (a call's time then runs to the start of the next call) for the roofline of the dominant
    # kernel; these events cost a little device time themselves and keep a call from being set up while its
    # predecessor drains, so the steps that carry them are a bit slower than the others - they are part of `value`.
    event_steps = min(args.steps, 3)
    ev = [[torch.cuda.Event(enable_timing=True) for _ in range(len(calls) + 1)] for _ in range(event_steps)]
    marks = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps + 1)]
    sampler = ClockSampler(local)
    sampler.start()
    time.sleep(0.25)
    barrier()
    t0 = time.time()
    marks[0].record(stream)
    for k in range(args.steps):
        step(ev[k] if k < event_steps else None)
        marks[k + 1].record(stream)
    barrier()
    t1 = time.time()
    total_ms = marks[0].elapsed_time(marks[args.steps])
    step_ms = [marks[k].elapsed_time(marks[k + 1]) for k in range(args.steps)]
    # keep the GPU under the same load a little longer so the clock sampler sees it
    if t1 - t0 < 0.6:
        tend = time.time() + 0.6
        while time.time() < tend:
            step()
        torch.cuda.synchronize()
        t1 = time.time()
    clocks = sampler.stop(t0, t1)
    total_ms = max_over_ranks(total_ms)
    ms_per_step = total_ms / args.steps
    value = whole_job_gbs(bytes_per_step, world, ms_per_step)
    plain_steps = step_ms[event_steps:] or step_ms
    check_status()

    # ---- the same step replayed from a CUDA graph (spares the launch gaps; reported beside `value`) ----
    graph_rec = None
    if not args.no_graph and args.op == "fused":
        try:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                step()
            graph.replay()
            check_status()
            g0, g1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            g0.record(stream)
            for _ in range(5):
                graph.replay()
            g1.record(stream)
            torch.cuda.synchronize()
            g_ms = g0.elapsed_time(g1) / 5
            graph_rec = {"ms_per_step": g_ms, "value": whole_job_gbs(bytes_per_step, 1, g_ms), "unit": UNIT,
                         "steps": 5, "note": "the step captured once and replayed; this rank only"}
            del graph
        except Exception as err:       # noqa: BLE001
            graph_rec = {"unavailable": str(err)[:200]}
            torch.cuda.synchronize()

    # ---- per-call device times inside the timed region -> roofline of the dominant kernel ----
    per_call_ms = [statistics.mean(ev[k][ci].elapsed_time(ev[k][ci + 1]) for k in range(event_steps))
                   for ci in range(len(calls))]
    # dominant kernel: the resident form of the column walk
    def resident(shape):
        form = b.team_geometry(b.F32, shape)
        return form is not None and form["taken"] == 1

    dominant = [ci for ci, (i, _) in enumerate(calls) if plans[ci][0] == b.PLAN_COLWALK and resident(specs[i].shape)]
    dom_bytes = sum(specs[calls[ci][0]].numel for ci in dominant) * bpe
    dom_ms = sum(per_call_ms[ci] for ci in dominant)
    achieved = dom_bytes / (dom_ms * 1e-3) / 1e9 if dominant else None
    rec = recorded_traffic()
    roofline = {
        "bound": "hbm", "kernel": "colteam_lag_kernel<float>",
        "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": (achieved / peak) if achieved else None,
        "peak_source": peak_src, "frac_of_nominal_8TBs": (achieved / NOMINAL_HBM_GBS) if achieved else None,
        "launches_per_step": len(dominant),
        "avg_launch_ms": dom_ms / max(1, len(dominant)),
        "avg_algorithmic_bytes_per_launch": dom_bytes / max(1, len(dominant)),
        "traffic": (rec["dram_bytes_per_algorithmic_byte"] * dom_bytes / max(1, len(dominant)) if rec else None),
        "traffic_source": (rec["source"] if rec else None),
        "share_of_step_time": dom_ms / sum(per_call_ms),
        "note": "achieved = algorithmic bytes of the launches / their CUDA-event time (from the event before a call to the event before the next: launch gaps included; events in the first 3 timed steps)",
    }
    in_step = []
    for ci, (i, bits) in enumerate(calls):
        gbs = specs[i].numel * bpe / (per_call_ms[ci] * 1e-3) / 1e9
        in_step.append({"tensor": specs[i].name, "bits": bits, "us": round(per_call_ms[ci] * 1e3, 2),
                        "GBps": round(gbs, 1), "frac_measured": round(gbs / peak, 3), "plan": plans[ci][0]})

    # ---- helpers for the bounded records below ----
    def sustained_us(run, n_calls, reps=3):
        """Median and best time per call of `run(k)` for k in range(n_calls), launched back to back with no
        event between the calls."""
        run_all = lambda: [run(k) for k in range(n_calls)]      # noqa: E731
        run_all()
        torch.cuda.synchronize()
        ts = []
        for _ in range(reps):
            a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a0.record(stream)
            run_all()
            a1.record(stream)
            torch.cuda.synchronize()
            ts.append(a0.elapsed_time(a1) * 1e3 / n_calls)
        return statistics.median(ts), min(ts)

    def rotating(x, gy, groups, group=b.GROUP_CHANNEL, min_bytes=400_000_000):
        """Copies of (x, gy, outputs) whose four arrays together exceed three times the L2: calls that walk
        over them find their tensor cold.  A tensor that large by itself is its own single copy."""
        n = max(1, -(-min_bytes // (4 * x.numel() * x.element_size())))
        sets = [(x, gy, outputs_for(x, groups, group))]
        for _ in range(n - 1):
            sets.append((x.clone(), gy.clone(), outputs_for(x, groups, group)))
        return sets

    def frac(elems, bytes_per_elem, us):
        return elems * bytes_per_elem / us / 1e3 / peak

    per_tensor, per_bits, sub = [], {}, {}
    if not args.no_sub and args.op == "fused":
        # ---- every call of the step by itself: sustained, cold, no event between calls ----
        for i, s in enumerate(specs):
            x, gy, _ = dev[i]
            sets = rotating(x, gy, s.shape[1])
            n_calls = max(4, 2 * len(sets))
            for bits in s.bits:
                med, best = sustained_us(lambda k: one_call(*sets[k % len(sets)], bits), n_calls)
                per_tensor.append({"tensor": s.name, "bits": bits, "us": round(med, 2), "best_us": round(best, 2),
                                   "GBps": round(s.numel * 16 / med / 1e3, 1), "frac_measured": round(frac(s.numel, 16, med), 3),
                                   "frac_8TBs": round(s.numel * 16 / med / 1e3 / NOMINAL_HBM_GBS, 3),
                                   "elements_per_s": s.numel / (med * 1e-6), "copies": len(sets),
                                   "plan": b.fused_plan(b.F32, s.shape, flags=plan_flags)[0]})
                acc = per_bits.setdefault(bits, [0, 0.0])
                acc[0] += s.numel
                acc[1] += med
            del sets
        check_status()

        # ---- other group mode, plan, contract on tensors of the step ----
        def pick(name):
            for i, s in enumerate(specs):
                if name in s.name:
                    return i, s
            return None, None
        for name in ("cfg3.2", "cfg3.4"):
            i, s = pick(name)
            if s is None:
                continue
            x, gy, _ = dev[i]
            G = b.num_groups(s.shape, 1, b.GROUP_SAMPLE_CHANNEL)
            sets = rotating(x, gy, G, b.GROUP_SAMPLE_CHANNEL)
            med, best = sustained_us(lambda k: one_call(*sets[k % len(sets)], 4, group=b.GROUP_SAMPLE_CHANNEL),
                                     max(4, 2 * len(sets)))
            sub.setdefault("per_sample_groups", []).append(
                {"tensor": s.name, "groups": G, "us": round(med, 2), "frac_measured": round(frac(s.numel, 16, med), 3),
                 "plan": b.fused_plan(b.F32, s.shape, group=b.GROUP_SAMPLE_CHANNEL)[0]})
            del sets
        i, s = pick("cfg3.4")
        if s is not None:          # the 'conventional' per-channel loop: three launches per channel
            x, gy, out = dev[i]
            med, best = sustained_us(lambda k: one_call(x, gy, out, 4, fl=b.FLAG_FORCE_NAIVE), 2, reps=2)
            sub["naive_per_channel_loop"] = [{"tensor": s.name, "launches": 3 * s.shape[1], "us": round(med, 1),
                                              "frac_measured": round(frac(s.numel, 16, med), 4)}]
        # default contract: every call clears its own workspace (no GRANQ_FLAG_WORKSPACE_ZEROED)
        for _ in range(2):
            for ci, (i, bits) in enumerate(calls):
                one_call(*dev[i], bits, fl=plan_flags)
        d0, d1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        d0.record(stream)
        for _ in range(3):
            for ci, (i, bits) in enumerate(calls):
                one_call(*dev[i], bits, fl=plan_flags)
        d1.record(stream)
        torch.cuda.synchronize()
        d_ms = d0.elapsed_time(d1) / 3
        sub["default_workspace_contract"] = {"ms_per_step": d_ms, "value": whole_job_gbs(bytes_per_step, 1, d_ms),
                                             "frac_measured": whole_job_gbs(bytes_per_step, 1, d_ms) / peak,
                                             "note": "every call clears its workspace itself (one memset node more "
                                                     "per call); 3 eager steps"}
        check_status()

        if rank == 0 and not args.only:
            # ---- configs 1, 2, 5 (bounded: a few calls each) ----
            s1 = wl.config_tensors(1)[0]
            x1 = torch.from_numpy(wl.make_activation(s1)).cuda()
            g1_ = torch.from_numpy(wl.make_upstream_grad(s1)).cuda()
            sets = rotating(x1, g1_, s1.shape[1])
            cold, _ = sustained_us(lambda k: one_call(*sets[k % len(sets)], 3), len(sets))
            warm, _ = sustained_us(lambda k: one_call(*sets[0], 3), 50)
            sub["config1"] = {"tensor": s1.name, "bits": 3, "cold_us": round(cold, 2), "warm_us": round(warm, 2),
                              "cold_frac_measured": round(frac(s1.numel, 16, cold), 4),
                              "warm_frac_measured": round(frac(s1.numel, 16, warm), 4),
                              "note": "1 MB tensor: launch-bound (the host needs about 10 us per call)"}
            del sets
            c2 = wl.config_tensors(2)
            t2 = []
            for s in c2:
                x = torch.from_numpy(wl.make_activation(s)).cuda()
                gy = torch.from_numpy(wl.make_upstream_grad(s)).cuda()
                t2.append((x, gy, outputs_for(x, s.shape[1])))
            calls2 = [(j, bits) for bits in (3, 4) for j in range(len(c2))]
            e2 = sum(c2[j].numel for j, _ in calls2)
            cold, _ = sustained_us(lambda k: one_call(*t2[calls2[k][0]], calls2[k][1]), len(calls2))
            small = [j for j, s in enumerate(c2) if s.shape[1] == 64][:2]       # 2 x 4 x 4.2 MB: stays in the L2
            warm, _ = sustained_us(lambda k: one_call(*t2[small[k % 2]], 3), 40)
            # the same 38 tensors through ONE host call (granq_fakequant_fused_batch: descriptors marshalled once)
            batch2 = b.FusedBatch([(t2[j][0], bits, t2[j][1]) for j, bits in calls2], outs=[t2[j][2] for j, _ in calls2],
                                  zeroed=True)
            bat, _ = sustained_us(lambda k: batch2.run(stream=stream), 1)
            sub["config2"] = {"calls": len(calls2), "elements": e2, "ms_per_set": cold * len(calls2) / 1e3,
                              "cold_frac_measured": round(frac(e2, 16, cold * len(calls2)), 3),
                              "batched_ms_per_set": bat / 1e3, "batched_frac_measured": round(frac(e2, 16, bat), 3),
                              "warm_small_tensor_us": round(warm, 2),
                              "warm_small_tensor_frac_measured": round(frac(c2[small[0]].numel, 16, warm), 3),
                              "note": "19 tensors x b in {3,4}, 772 MB working set (cold between calls); batched = the "
                                      "38 calls as one granq_fakequant_fused_batch call (the host's per-call cost gone); "
                                      "the 4 MB tensors alternating in pairs stay in the L2 (warm) and are launch-bound"}
            del t2
            torch.cuda.empty_cache()
            gen = torch.Generator(device="cuda").manual_seed(5000)
            rows5 = []
            for s in wl.config_tensors(5):
                # values of the same recipe generated on the device (Student-t(3), per-channel log-normal spread)
                sig = torch.exp(torch.randn(1, s.shape[1], 1, 1, device="cuda", generator=gen))
                x32 = torch.randn(s.shape, device="cuda", generator=gen)
                den = torch.zeros(s.shape, device="cuda")
                for _ in range(3):
                    den += torch.randn(s.shape, device="cuda", generator=gen) ** 2
                x32 = x32 / torch.sqrt(den / 3.0).clamp_min(1e-6) * sig
                del den
                g32 = torch.randn(s.shape, device="cuda", generator=gen)
                for dt in ("f32", "bf16"):
                    x = x32 if dt == "f32" else x32.bfloat16()
                    gy = g32 if dt == "f32" else g32.bfloat16()
                    out = outputs_for(x, s.shape[1])
                    e = x.element_size()
                    fused, _ = sustained_us(lambda k: one_call(x, gy, out, 2 + k % 7), 7, reps=2)
                    fwd, _ = sustained_us(lambda k: one_call(x, None, out, 2 + k % 7, op="fused_fwd"), 7, reps=2)
                    rows5.append({"tensor": s.name, "dtype": dt, "bits": "2..8 (one call each)",
                                  "fused_us": round(fused, 1), "fused_frac_measured": round(frac(s.numel, 4 * e, fused), 3),
                                  "fwd_only_us": round(fwd, 1), "fwd_only_frac_measured": round(frac(s.numel, 2 * e, fwd), 3),
                                  "elements_per_s_fused": s.numel / (fused * 1e-6),
                                  "plan": b.fused_plan(b.F32 if dt == "f32" else b.BF16, s.shape)[0]})
                    del out
                del x32, g32
                torch.cuda.empty_cache()
            sub["config5"] = {"rows": rows5, "data": "device-generated Student-t(3) x per-channel log-normal spread "
                                                     "(same recipe as the parity inputs); each tensor is larger "
                                                     "than the L2, so every call is cold"}

        if rank == 0 and not args.only:
            # ---- the other entry points over the step's tensors (one pass each, b = 4) ----
            for x, gy, out in dev:
                out.packed_mask = b.make_packed_mask(x)
                one_call(x, gy, out, 4)          # a range for the calls that take one
            rows = {}
            for op, bytes_pe in (("range", 4), ("fwd", 8), ("bwd", 12), ("fused_fwd", 8), ("fused_fwd_packmask", 8.125),
                                 ("bwd_packmask", 8.125)):
                med, _ = sustained_us(lambda k: one_call(*dev[k], 4, op=op), len(dev), reps=2)
                tot = sum(s.numel for s in specs)
                big = [i for i, s in enumerate(specs) if s.numel * 4 >= 100_000_000]
                med_big, _ = sustained_us(lambda k: one_call(*dev[big[k]], 4, op=op), len(big), reps=2)
                rows[op] = {"bytes_per_element": bytes_pe, "frac_measured_all_12": round(frac(tot, bytes_pe, med * len(dev)), 3),
                            "frac_measured_100MB_and_up": round(frac(sum(specs[i].numel for i in big), bytes_pe,
                                                                     med_big * len(big)), 3)}
            sub["entry_points"] = rows
            check_status()
            # ---- packed integer codes on one tensor (4 + b/8 bytes per element each way) ----
            rows = []
            for name, bits in (("cfg3.1", 3), ("cfg3.1", 4), ("cfg3.1", 5), ("cfg4.6", 4)):      # the last one: 7x7 planes
                i, s = pick(name)
                x, gy, out = dev[i]
                pc = torch.empty(b.packed_codes_bytes(x.shape, bits) // 4, dtype=torch.int32, device="cuda")
                q = b.granq_quantize_packed(x, bits, out.lo, out.hi, packed_codes=pc, stream=stream)
                tq, _ = sustained_us(lambda k: b.granq_quantize_packed(x, bits, out.lo, out.hi, packed_codes=pc,
                                                                       stream=stream), 3, reps=2)
                td, _ = sustained_us(lambda k: b.granq_dequantize_packed(pc, x.shape, x.dtype, bits, q.s, q.z, y=out.y,
                                                                         stream=stream), 3, reps=2)
                fo = b.granq_quantize_packed_fused(x, bits, packed_codes=pc, stream=stream)
                tf, _ = sustained_us(lambda k: b.granq_quantize_packed_fused(x, bits, out=fo, stream=stream), 3, reps=2)
                rows.append({"tensor": s.name, "bits": bits, "quantize_us": round(tq, 1),
                             "quantize_frac_measured": round(frac(s.numel, 4 + bits / 8, tq), 3),
                             "fused_range_and_quantize_us": round(tf, 1),
                             "fused_frac_measured": round(frac(s.numel, 4 + bits / 8, tf), 3),
                             "dequantize_us": round(td, 1), "dequantize_frac_measured": round(frac(s.numel, 4 + bits / 8, td), 3)})
            sub["packed_codes"] = rows
            # ---- the accumulation over the codes on the tensor cores (Eq. 6 left-hand side, pointwise case) ----
            rows = []
            for name, oc in (("cfg3.1", 64), ("cfg3.3", 256)):
                i, s = pick(name)
                x, gy, out = dev[i]
                qp = b.granq_quantize_packed(x, 4, out.lo, out.hi, stream=stream)
                wt = torch.randn(oc, s.shape[1], device="cuda") / 8
                ya, wsa = b.granq_accumulate_codes(qp.packed_codes, s.shape, 4, qp.s, qp.z, wt, stream=stream)
                ta, _ = sustained_us(lambda k: b.granq_accumulate_codes(qp.packed_codes, s.shape, 4, qp.s, qp.z, wt, y=ya,
                                                                        workspace=wsa, stream=stream), 3, reps=2)
                assert b.workspace_status(wsa) == b.OK
                pix = s.numel // s.shape[1]
                alg = s.numel * 0.5 + pix * oc * 4 + oc * s.shape[1] * 4          # packed codes in, y out, weights in
                flops = 2.0 * pix * s.shape[1] * oc * 2                          # two bf16 halves of the weights
                rows.append({"tensor": s.name, "out_channels": oc, "us": round(ta, 1),
                             "frac_measured_hbm": round(alg / ta / 1e3 / peak, 3), "tflops": round(flops / ta / 1e6, 1),
                             "note": "two launches: weights (scale folded in, hi / lo halves, bias), then code expansion + contraction + epilogue in one persistent kernel"})
            sub["accumulate_codes"] = rows
            # ---- all weight tensors of a network in one launch against one fused call per tensor ----
            rows = []
            for net in ("resnet20", "resnet18"):
                ws = [torch.from_numpy(w).cuda() for w in wl.make_weights(net)]
                gs = [torch.from_numpy(g).cuda() for g in wl.make_weights(net, grads=True)]
                ws4 = [w.reshape(w.shape[0], -1, 1, 1) for w in ws]
                gs4 = [g.reshape(g.shape[0], -1, 1, 1) for g in gs]
                wouts = [b.FakeQuantOut(y=torch.empty_like(w), gx=torch.empty_like(w), workspace=b.make_workspace(w, 0))
                         for w in ws4]
                batch = b.WeightBatch(ws, 4, grads=gs)
                tb, _ = sustained_us(lambda k: batch.run(stream=stream), 5)
                tl, _ = sustained_us(lambda k: b.granq_fakequant_fused(ws4[k], 4, gy=gs4[k], channel_axis=0, out=wouts[k],
                                                                       stream=stream), len(ws4))
                rows.append({"network": net, "tensors": len(ws), "elements": sum(w.numel() for w in ws),
                             "batched_us": round(tb, 1), "one_call_per_tensor_us": round(tl * len(ws4), 1)})
            sub["weights"] = rows
            # ---- Table 2 in kind: layer-wise against channel-wise at 3 bits on the ResNet-20-shaped set ----
            rows, seen = [], set()
            for s2 in wl.config_tensors(2):
                if s2.shape in seen:
                    continue
                seen.add(s2.shape)
                x2 = torch.from_numpy(wl.make_activation(s2)).cuda()
                row = {"tensor": s2.name, "bits": 3}
                for name, group in (("layer_wise", b.GROUP_TENSOR), ("channel_wise", b.GROUP_CHANNEL)):
                    o2 = b.FakeQuantOut(y=torch.empty_like(x2))
                    b.granq_fakequant_fused_stats(x2, 3, group=group, out=o2, stream=stream)
                    torch.cuda.synchronize()
                    cos, rel = b.distortion_from_sums(o2.sums.cpu().tolist())
                    row[name] = {"cosine": round(cos, 4), "rel_error": round(rel, 4)}
                rows.append(row)
                del x2
            sub["table2_in_kind"] = {"rows": rows, "paper": "ResNet-20, 3 bits: layer-wise 0.5111 / 0.3129, channel-wise "
                                                            "0.6835 / 0.1063 (cosine / relative error; other data)"}
            # ---- Table 5 in kind: one forward pass over the 19 ResNet-20 activation tensors at batch 16, 3 bits ----
            import dataclasses
            s16 = [dataclasses.replace(s2, shape=(16,) + tuple(s2.shape[1:])) for s2 in wl.config_tensors(2)]
            x16 = [torch.from_numpy(wl.make_activation(s2)).cuda() for s2 in s16]
            rows = []
            for name, group, fl in (("layer-wise", b.GROUP_TENSOR, 0),
                                    ("channel-wise, per-channel loop", b.GROUP_CHANNEL, b.FLAG_FORCE_NAIVE),
                                    ("channel-wise, default plan", b.GROUP_CHANNEL, 0)):
                o16 = [b.FakeQuantOut(y=torch.empty_like(x), workspace=b.make_workspace(x, 1, group)) for x in x16]
                launches = sum(b.fused_plan(b.F32, x.shape, group=group, with_backward=False, flags=fl)[1] for x in x16)

                def one_pass():
                    for x, o in zip(x16, o16):
                        b.granq_fakequant_fused(x, 3, group=group, out=o, flags=fl, stream=stream)
                one_pass()
                torch.cuda.synchronize()
                walls = []
                for _ in range(5):
                    w0 = time.perf_counter()
                    one_pass()
                    torch.cuda.synchronize()
                    walls.append((time.perf_counter() - w0) * 1e3)
                rows.append({"scheme": name, "ms_per_pass_wall": round(statistics.median(walls), 3), "launches": launches})
            sub["table5_in_kind"] = {"rows": rows, "paper_ms": {"layer-wise": 0.227, "channel-wise (conventional)": 103.671,
                                                                "GranQ": 0.236}, "paper_hardware": "not stated"}

    sharded = None
    if args.sharded:
        from paper_2503_18339_b200 import data_parallel as dp
        for x, gy, out in dev:
            out.packed_mask = b.make_packed_mask(x)

        def sharded_step():
            for i, bits in calls:
                x, gy, out = dev[i]
                lo, hi = b.granq_range(x, lo=out.lo, hi=out.hi, workspace=out.workspace, stream=stream)
                dp.sync_range(lo, hi, stream=stream)
                b.granq_fakequant_fwd_packmask(x, bits, lo, hi, y=out.y, packed_mask=out.packed_mask, stream=stream)
                b.granq_fakequant_bwd_packmask(gy, out.packed_mask, gx=out.gx, stream=stream)
        sharded_step()
        barrier()
        h0, h1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        h0.record(stream)
        for _ in range(3):
            sharded_step()
        h1.record(stream)
        barrier()
        h_ms = max_over_ranks(h0.elapsed_time(h1) / 3)
        sharded = {"ms_per_step": h_ms, "value": whole_job_gbs(int(elems_per_step * 20.25), world, h_ms), "unit": UNIT,
                   "bytes_per_element": 20.25, "scaling": "strong in the batch: every rank holds 1/N of a global batch "
                   "and all ranks quantize with its range",
                   "note": "range (4 B) + all-reduce of 2*C floats + forward with packed mask (8.125 B) + backward "
                           "from the mask (8.125 B)"}

    # ---- end to end through the host-buffer entry point (pinned memory, copies timed) ----
    e2e = None
    if args.e2e_steps > 0:
        # Two streams, each with its own arena and host result buffers: while one call's results go
        # down to the host the next call's inputs go up (PCIe is full duplex).
        big = max(specs, key=lambda s: s.numel)
        cmax = max(s.shape[1] for s in specs)
        lanes = []
        for _ in range(max(1, args.e2e_lanes)):
            lanes.append({
                "stream": torch.cuda.Stream(),
                "arena": torch.empty(b.host_arena_bytes(b.F32, big.shape), dtype=torch.uint8, device="cuda"),
                "y": torch.empty(big.shape, dtype=torch.float32).pin_memory(),
                "gx": torch.empty(big.shape, dtype=torch.float32).pin_memory(),
                "lo": torch.empty(cmax).pin_memory(), "hi": torch.empty(cmax).pin_memory(), "last": None})

        # both bit-widths of a tensor back to back, one per lane: the two lanes then move equal amounts at the
        # same time and one lane's download overlaps the other's upload best
        e2e_calls = [(i, bits) for i, sp in enumerate(specs) for bits in sp.bits]

        def e2e_step():
            for k, (i, bits) in enumerate(e2e_calls):
                ln = lanes[k % len(lanes)]
                xs, gs = host[i]
                n, c = specs[i].numel, specs[i].shape[1]
                b.granq_fakequant_fused_host(xs, bits, gs, ln["y"].view(-1)[:n].view(specs[i].shape),
                                             ln["gx"].view(-1)[:n].view(specs[i].shape), ln["lo"][:c], ln["hi"][:c],
                                             ln["arena"], flags=b.FLAG_HOST_ASYNC, stream=ln["stream"])
                ln["last"] = specs[i].shape

        def e2e_fence(check):
            for ln in lanes:
                stream.wait_stream(ln["stream"])
                if check:
                    assert b.host_arena_status(b.F32, ln["last"], ln["arena"], stream=ln["stream"]) == b.OK

        for ln in lanes:
            ln["stream"].wait_stream(stream)
        e2e_step()
        e2e_fence(True)
        barrier()
        a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a0.record(stream)
        for ln in lanes:
            ln["stream"].wait_stream(stream)
        for _ in range(args.e2e_steps):
            e2e_step()
        e2e_fence(False)
        a1.record(stream)
        barrier()
        e2e_fence(True)
        e_ms = a0.elapsed_time(a1)
        e_ms = max_over_ranks(e_ms)
        e2e = {"value": whole_job_gbs(bytes_per_step, world, e_ms / args.e2e_steps), "unit": UNIT,
               "h2d_bytes_per_step": elems_per_step * 8, "d2h_bytes_per_step": elems_per_step * 8 +
               sum(specs[i].shape[1] * 8 for i, _ in calls),
               "steps": args.e2e_steps, "ms_per_step": e_ms / args.e2e_steps,
               "api": ("granq_fakequant_fused_host (pinned host buffers; calls rotate over %d streams and arenas, "
                       "so one call's downloads overlap the next call's uploads)" % len(lanes))}

    # ---- the CPU oracle on a bounded sample, rank 0 at N = 1 only ----
    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        arrays = {sp.name: (xs.numpy(), gs.numpy()) for sp, (xs, gs) in zip(specs, host)}
        sample = [(specs[i], bits) for i, bits in calls if specs[i].numel <= 60_000_000]
        s, e = time_oracle(sample, arrays)
        repeats = max(1, min(8, int(10.0 / max(s, 1e-3))))        # about 10 s of CPU work in all
        for _ in range(repeats - 1):
            s2, e2 = time_oracle(sample, arrays)
            s, e = s + s2, e + e2
        # the same oracle calls spread over the host's cores (one call per thread at a time; ctypes releases the GIL)
        from concurrent.futures import ThreadPoolExecutor
        from oracle import granq_oracle as orc
        threads = max(1, min(os.cpu_count() or 1, len(sample)))
        tp0 = time.perf_counter()
        with ThreadPoolExecutor(max_workers=threads) as pool:
            list(pool.map(lambda sb: orc.fused(arrays[sb[0].name][0], sb[1], gy=arrays[sb[0].name][1], want_codes=False),
                          sample))
        tp = time.perf_counter() - tp0
        par_elems = sum(sp.numel for sp, _ in sample)
        cpu = {"value": e * BYTES_PER_ELEM / s / 1e9, "unit": UNIT, "cores": 1, "kind": "oracle",
               "all_cores": {"value": par_elems * BYTES_PER_ELEM / tp / 1e9, "unit": UNIT, "threads": threads,
                             "how": "the sample's calls once over, one oracle call per thread at a time"},
               "sample": "every workload tensor of at most 60 M elements, b=4 and b=5 (%d calls), %d times over: %d M elements"
                         % (len(sample), repeats, e // 1_000_000), "seconds": round(s, 2), "elements_per_s": e / s,
               "host_cores_available": os.cpu_count()}

    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps, "warmup": warmup,
            "ms_per_step": ms_per_step, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32", "data": "synthetic",
            "config": {"workload": WORKLOAD, "elements_per_step_per_gpu": elems_per_step,
                       "calls_per_step": len(calls),
                       "l2": "inputs larger than L2: a step is all 12 tensors at 4 bits, then all 12 at 5 bits, so "
                             "3.6 GB pass through the 126 MB L2 between two calls on the same tensor (every call is cold)",
                       "group_mode": "channel",
                       "launch": ("every step launched eagerly through the C ABI; steps 1..%d carry one CUDA event per "
                                  "call" % event_steps),
                       "workspace": ("cleared by every call" if args.clear_workspace else
                                     "cleared once at allocation, GRANQ_FLAG_WORKSPACE_ZEROED on every call"),
                       "parallelism": f"replicas x{world} (independent batches, no exchange)"},
            "step_ms": {"mean": ms_per_step, "median": statistics.median(step_ms), "best": min(step_ms),
                        "median_without_call_events": statistics.median(plain_steps), "rank": 0},
            "value_median_step": whole_job_gbs(bytes_per_step, world, statistics.median(step_ms)),
            "value_best_step": whole_job_gbs(bytes_per_step, world, min(step_ms)),
            "elements_per_s": world * elems_per_step / (ms_per_step * 1e-3),
            "elements_per_s_by_bits": {str(k): v[0] / (v[1] * 1e-6) for k, v in sorted(per_bits.items())},
            "frac_of_measured_hbm": value / world / peak, "frac_of_nominal_8TBs": value / world / NOMINAL_HBM_GBS,
            "gpu_launches": launches_per_step * args.steps, "clocks": clocks, "e2e": e2e, "roofline": roofline,
            "cpu_baseline": cpu, "graph_replay": graph_rec, "per_tensor": per_tensor, "in_step": in_step, "sub": sub,
            "sharded": sharded,
        }
        print(json.dumps(line))
        if args.table:
            for r in (per_tensor or in_step):
                print(f"{r['tensor']:28s} b={r['bits']} {r['us']:9.1f} us {r['GBps']:8.1f} GB/s "
                      f"{100 * r['frac_measured']:5.1f}% of measured plan {r['plan']}", file=sys.stderr)
    if world > 1:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
