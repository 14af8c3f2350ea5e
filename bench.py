#!/usr/bin/env python
"""Benchmark of the shard-elastic execution path on B200.

One step = one forward of the whole path over one batch: every layer's shard decode fused into
its four GEMMs, attention, residual+LayerNorm, and (end-to-end arm) the layerwise streaming of
shards from pinned host memory behind compute.

Workload at N=1: configuration 4 of the benchmark list - 24-layer BERT-large, batch 1, seq 256,
all units kept, per-unit bitwidths 2-6 skewed toward 3.
  value : packed-weight GB/s with every shard resident in device memory before the timed region
  e2e   : the same metric through sti_model_forward_host - x from pinned host memory, layers 2..23
          streamed host-to-device during execution behind a 2-layer preload buffer, y copied back
N>1 runs one independent replica per GPU (the path has no exchange step): weak scaling.

`--impl reference` times the CPU oracle (the deliberately plain numpy implementation) instead.
"""
from __future__ import annotations

import argparse
import dataclasses
import json
import os
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

METRIC = "packed_weight_GBps"
UNIT = "GB/s"
WORKLOAD = ("24-layer BERT-large (hidden 1024, 16 heads x 64, FFN 4096 in 16 slices), batch 1, "
            "seq 256, all shard units kept, bits ~ {2:.15,3:.45,4:.20,5:.10,6:.10}")
FALLBACK_PEAKS = {"hbm_gbs": 6650.0, "bf16_tflops": 1590.0, "bf16_tflops_sustained": 1400.0}


# dram__bytes_read.sum + dram__bytes_write.sum per dequant-GEMM launch (mean over one layer's QKV, O, FFN1, FFN2
# launches; BERT-large layer, batch 1, seq 256) from an ncu --set full capture of the present dqgemm.cu.
NCU_DRAM_BYTES_PER_GEMM_LAUNCH = 2522368


def load_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as fh:
            return json.load(fh), "of measured (MEASURED_PEAKS.json)"
    return dict(FALLBACK_PEAKS), "of fallback"


def gemm_flops(work) -> float:
    sh, T = work.shape, work.batch * work.seq
    total = 0.0
    for l in range(sh.n_layers):
        nh, ns = len(work.kept(l, 0)), len(work.kept(l, 1))
        total += 2.0 * T * (4 * sh.hidden * sh.head_dim * nh + 2 * sh.hidden * sh.slice_width * ns)
    return total


def attn_flops(work) -> float:
    sh = work.shape
    return sum(4.0 * work.batch * work.seq ** 2 * sh.head_dim * len(work.kept(l, 0)) for l in range(sh.n_layers))


def with_residency(work, resident_layers: int):
    import workloads as W
    attn = [[W.UnitPlan(u.keep, u.bits, l < resident_layers) for u in layer] for l, layer in enumerate(work.attn_plan)]
    ffn = [[W.UnitPlan(u.keep, u.bits, l < resident_layers) for u in layer] for l, layer in enumerate(work.ffn_plan)]
    return dataclasses.replace(work, attn_plan=attn, ffn_plan=ffn)


class ClockSampler:
    """nvidia-smi clocks and throttle reasons while the timed regions run."""
    QUERY = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.QUERY}",
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except OSError:
            self.proc = None

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
        sm, smax, power, reasons = [], [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 8:
                continue
            try:
                sm.append(float(parts[0])); smax.append(float(parts[1])); power.append(float(parts[2]))
            except ValueError:
                continue
            for name, val in zip(names, parts[4:8]):
                if val.lower().startswith("active"):
                    reasons.add(name)
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "power_w_max": max(power) if power else None, "samples": len(sm), "reasons": sorted(reasons)}


def max_over_ranks(local_ms: float, world: int, device: str = "cuda") -> float:
    """Timing rule for N > 1: every rank times its own replica on its device, the job's time is the slowest rank's."""
    if world <= 1:
        return float(local_ms)
    import torch
    import torch.distributed as dist
    t = torch.tensor([local_ms], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def aggregate_throughput(units_per_rank: float, world: int, ms_per_step: float) -> float:
    """Whole-job throughput of `world` independent replicas (weak scaling): all ranks' units over the slowest time."""
    return units_per_rank * world / (ms_per_step * 1e-3)


def oracle_forward_timed(work, layers):
    from oracle import sti_oracle as O
    t0 = time.perf_counter()
    O.run_workload(work, layers=layers)
    return time.perf_counter() - t0


def blas_threads() -> int:
    try:
        from threadpoolctl import threadpool_info
        n = [p.get("num_threads", 1) for p in threadpool_info() if p.get("user_api") == "blas"]
        return max(n) if n else (os.cpu_count() or 1)
    except Exception:
        return os.cpu_count() or 1


def run_reference(args):
    """The CPU oracle as it stands, on the same workload and metric (bounded sample per step)."""
    if int(os.environ.get("RANK", "0")) != 0:
        return
    import workloads as W
    work = W.make_config(4, workers=min(8, os.cpu_count() or 1))
    n_sample = work.shape.n_layers                 # the whole model: the same configuration as the GPU arm
    layers = list(range(n_sample))
    for _ in range(args.warmup):
        oracle_forward_timed(work, layers)
    total = sum(oracle_forward_timed(work, layers) for _ in range(args.steps))
    value = work.packed_bytes() * args.steps / total / 1e9
    sample = f"all {n_sample} layers (decode + fp64 forward, 1 sequence of 256 tokens) per step"
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": total / args.steps * 1e3,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": WORKLOAD, "sample": sample},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": blas_threads(), "kind": "oracle", "sample": sample},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        "gpu_launches": 0,
    }))


def device_act(torch, work):
    if work.act_dtype == "bf16":
        return torch.from_numpy(work.x_dev.view(np.int16).copy()).cuda().view(torch.bfloat16)
    return torch.from_numpy(work.x_dev).cuda()


def time_layer_config(sti, torch, number, peaks, iters=60, seq=None):
    """Cold-L2 latency of one sti_layer_forward on configuration 1 or 2 (microseconds); `seq` shortens the
    sequence for the weight-streaming probe shapes (few tokens: the GEMMs are HBM-bound by the roofline)."""
    import workloads as W
    work = W.make_config(number, seq=seq)
    stream = torch.cuda.Stream()
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    times = []
    with sti.Session(work, compute_stream=stream.cuda_stream) as s:
        x = device_act(torch, work)
        y = torch.empty_like(x)
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            for i in range(iters + 5):
                flush.zero_()
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                sti.sti_layer_forward(s.plan, 0, x.data_ptr(), y.data_ptr(), work.batch, work.seq)
                e1.record(stream)
                stream.synchronize()
                if i >= 5:
                    times.append(e0.elapsed_time(e1) * 1e3)
        sti.sti_sync(s.ctx)
    packed = work.packed_bytes()
    flops = gemm_flops(work) + attn_flops(work)
    act = 2 * work.x_dev.nbytes
    floor_us = max((packed + act) / (peaks["hbm_gbs"] * 1e9), flops / (peaks["bf16_tflops_sustained"] * 1e12)) * 1e6
    med = float(np.median(times))
    t_hbm = (packed + act) / (peaks["hbm_gbs"] * 1e9) * 1e6
    return {"tokens": work.batch * work.seq, "bound": "hbm" if t_hbm >= floor_us * 0.999 else "tensor",
            "packed_frac_of_hbm_peak": packed / med / 1e3 / peaks["hbm_gbs"],
            "layer_us_median": med, "layer_us_p10": float(np.percentile(times, 10)),
            "layer_us_p90": float(np.percentile(times, 90)), "packed_bytes": packed, "flops": flops,
            "packed_GBps": packed / med / 1e3, "roofline_floor_us": floor_us, "x_of_floor": med / floor_us,
            "l2": "flushed before every call"}


def run_sweep(args):
    """Configuration 5: BERT-large stack, batch {1,8,32,64} x seq {128,512}, uniform 3-bit and mixed 2-6-bit
    plans, shards resident vs streamed (2-layer preload).  Prints one JSON object with a row per point."""
    import workloads as W
    from workloads.shards import round_to_bf16
    n_layers = args.layers or 24
    works = {plan: W.make_config(5, n_layers=n_layers, plan=plan, resident=False, batch=1, seq=128,
                                 workers=min(8, os.cpu_count() or 1)) for plan in ("uniform3", "mixed")}
    import torch
    import paper_2207_05022_b200 as sti
    from paper_2207_05022_b200 import build
    build.build_library()
    peaks, peak_src = load_peaks()
    for k, v in FALLBACK_PEAKS.items():
        peaks.setdefault(k, v)
    stream = torch.cuda.Stream()
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    batches = [int(b) for b in args.sweep_batches.split(",")]
    seqs = [int(q) for q in args.sweep_seqs.split(",")]
    rows = []
    rng = np.random.default_rng(0)
    for plan, work in works.items():
        sessions = {"resident": sti.Session(with_residency(work, n_layers), compute_stream=stream.cuda_stream,
                                            max_batch=max(batches), max_seq=max(seqs)),
                    "streamed": sti.Session(work, compute_stream=stream.cuda_stream, max_batch=max(batches),
                                            max_seq=max(seqs))}
        packed = work.packed_bytes()
        for B in batches:
            for L in seqs:
                bits16, _ = round_to_bf16(rng.standard_normal((B, L, work.shape.hidden), dtype=np.float32))
                x = torch.from_numpy(bits16.view(np.int16)).cuda().view(torch.bfloat16)
                y = torch.empty_like(x)
                shaped = dataclasses.replace(work, batch=B, seq=L)
                flops_g, flops_a = gemm_flops(shaped), attn_flops(shaped)
                row = {"plan": plan, "batch": B, "seq": L, "tokens": B * L, "packed_bytes": packed}
                for name, sess in sessions.items():
                    ms = []
                    with torch.cuda.stream(stream):
                        for i in range(args.warmup + args.steps):
                            flush.zero_()
                            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                            e0.record(stream)
                            sti.sti_model_forward(sess.plan, x.data_ptr(), y.data_ptr(), B, L)
                            e1.record(stream)
                            stream.synchronize()
                            if i >= args.warmup:
                                ms.append(e0.elapsed_time(e1))
                    sti.sti_sync(sess.ctx)
                    row[f"ms_{name}"] = float(np.median(ms))
                sess = sessions["resident"]
                sti.sti_plan_set_profiling(sess.plan, 2)
                gemm_us = []
                with torch.cuda.stream(stream):
                    for i in range(3):
                        flush.zero_()
                        sti.sti_model_forward(sess.plan, x.data_ptr(), y.data_ptr(), B, L)
                        st = sti.sti_get_stats(sess.plan)
                        gemm_us.append(sum(st.gemm_us[:st.n_layers]))
                sti.sti_plan_set_profiling(sess.plan, 0)
                g_s = float(np.median(gemm_us)) * 1e-6
                t_res = row["ms_resident"] * 1e-3
                row.update({
                    "gemm_ms": g_s * 1e3, "gemm_TFLOPs": flops_g / g_s / 1e12,
                    "gemm_frac_of_tensor_peak": flops_g / g_s / 1e12 / peaks["bf16_tflops_sustained"],
                    "gemm_packed_GBps": packed / g_s / 1e9,
                    "e2e_TFLOPs_resident": (flops_g + flops_a) / t_res / 1e12,
                    "packed_GBps_resident": packed / t_res / 1e9,
                    "packed_GBps_streamed": packed / (row["ms_streamed"] * 1e-3) / 1e9,
                    "streamed_over_resident": row["ms_streamed"] / row["ms_resident"]})
                rows.append(row)
        for sess in sessions.values():
            sess.close()
    print(json.dumps({"sweep": "BERT-large stack, bf16 activations", "n_layers": n_layers,
                      "peak_source": peak_src, "rows": rows}))


def planner_profile(args, widths=None):
    """Section 5.2's two offline profiles on the device in use: T_io per stored version and T_comp per submodel
    width m (see run_planner).  Returns everything the plan-and-execute modes need."""
    import workloads as W
    B, L = args.planner_batch, args.planner_seq
    workers = min(8, os.cpu_count() or 1)
    N, M = 24, 16
    versions = (2, 3, 4, 5, 6, 32)
    ones = np.ones((1, M), np.uint8)
    shard_bytes = [W.make_planned(ones, ones * k, ones * 0, batch=B, seq=L).packed_bytes() // M for k in versions]
    widths = list(widths) if widths else list(range(1, M + 1))      # submodel widths measured (others interpolated)
    depth = 4
    ring = args.planner_ring
    full = np.ones((depth, M), np.uint8)
    stack = W.make_planned(full, full * 2, full, batch=B, seq=L, workers=workers, ring_slots=ring)
    stack6 = W.make_planned(full, full * 6, full, batch=B, seq=L, workers=workers, ring_slots=ring)

    def narrowed(m, streamed_from=None):
        """The 4-layer 2-bit stack with shards 0..m-1 kept; layers >= streamed_from leave the preload buffer."""
        def grid(g):
            return [[dataclasses.replace(u, keep=i < m, resident=streamed_from is None or l < streamed_from)
                     for i, u in enumerate(row)] for l, row in enumerate(g)]
        return dataclasses.replace(stack, attn_plan=grid(stack.attn_plan), ffn_plan=grid(stack.ffn_plan),
                                   blobs={k: v for k, v in stack.blobs.items() if k[2] < m})

    import torch
    import paper_2207_05022_b200 as sti
    from paper_2207_05022_b200 import build
    build.build_library()
    stream = torch.cuda.Stream()
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")

    def forward_ms(sess, work, x, y, steps, warmup=3):
        ms = []
        with torch.cuda.stream(stream):
            for i in range(warmup + steps):
                flush.zero_()
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                sti.sti_model_forward(sess.plan, x.data_ptr(), y.data_ptr(), work.batch, work.seq)
                e1.record(stream)
                stream.synchronize()
                if i >= warmup:
                    ms.append(e0.elapsed_time(e1))
        sti.sti_sync(sess.ctx)
        return float(np.median(ms))

    # T_io: the rate the pipeline's own layer copies reach (pinned host arena -> ring slot, measured by the
    # library around each copy while the layers compute), applied to each version's bytes
    probe = narrowed(M, streamed_from=1)
    rates = []
    with sti.Session(probe, compute_stream=stream.cuda_stream) as sess:
        x = device_act(torch, probe)
        y = torch.empty_like(x)
        forward_ms(sess, probe, x, y, 10, warmup=10)
        sti.sti_plan_set_profiling(sess.plan, 1)
        with torch.cuda.stream(stream):
            for _ in range(9):
                sti.sti_model_forward(sess.plan, x.data_ptr(), y.data_ptr(), B, L)
                st = sti.sti_get_stats(sess.plan)
                rates.append(sum(st.streamed_bytes[:st.n_layers]) / (sum(st.copy_us[:st.n_layers]) * 1e3))
        sti.sti_plan_set_profiling(sess.plan, 0)
    h2d_gbps = float(np.median(rates))
    t_io_us = [b / (h2d_gbps * 1e3) for b in shard_bytes]

    # T_comp(m): per-layer delay of a resident stack that keeps m shards per layer, interpolated over m,
    # plus the pipeline's per-layer cost measured on the streamed twin
    def stack_ms(work):
        with sti.Session(work, compute_stream=stream.cuda_stream) as sess:
            x = device_act(torch, work)
            y = torch.empty_like(x)
            return forward_ms(sess, work, x, y, 20)
    measured = [stack_ms(narrowed(m)) * 1e3 / depth for m in widths]
    t_comp16_6bit = stack_ms(stack6) * 1e3 / depth
    # the 4-shard stack with layers 1.. streamed: its copies are far shorter than its layers, so what it
    # takes longer than the resident stack is the per-layer cost of running inside the pipeline
    pipe_us = max(0.0, (stack_ms(narrowed(4, streamed_from=1)) * 1e3 - float(np.interp(4, widths, measured)) * depth)
                  / (depth - 1))
    t_comp_us = [0.0] + [float(np.interp(m, widths, measured)) + pipe_us for m in range(1, M + 1)]
    t_comp_us = list(np.maximum.accumulate(t_comp_us))
    return dict(W=W, sti=sti, torch=torch, stream=stream, flush=flush, forward_ms=forward_ms, B=B, L=L, N=N, M=M,
                workers=workers, versions=versions, shard_bytes=shard_bytes, ring=ring, h2d_gbps=h2d_gbps,
                t_io_us=t_io_us, t_comp_us=t_comp_us, pipe_us=pipe_us, measured=measured, t_comp16_6bit=t_comp16_6bit)


def run_planner(args):
    """Section 5 end to end: profile the device (T_io per version, T_comp per width m), let the library's
    two-stage planner pick (n, m), bitwidths and the preload prefix for each target latency, execute the
    plan streamed from pinned host memory and report how much of the copy time the pipeline hid.
    Shard importance is a seeded uniform table (the paper profiles it on a dev set)."""
    pf = planner_profile(args)
    W, sti, torch, stream, flush, forward_ms = pf["W"], pf["sti"], pf["torch"], pf["stream"], pf["flush"], pf["forward_ms"]
    B, L, N, M, workers, ring = pf["B"], pf["L"], pf["N"], pf["M"], pf["workers"], pf["ring"]
    shard_bytes, h2d_gbps, t_io_us, t_comp_us, pipe_us = pf["shard_bytes"], pf["h2d_gbps"], pf["t_io_us"], pf["t_comp_us"], pf["pipe_us"]
    measured, t_comp16_6bit = pf["measured"], pf["t_comp16_6bit"]
    importance = np.random.default_rng(np.random.SeedSequence([0, 77])).uniform(0, 1, (N, M)).astype(np.float32)
    preload_bytes = int(args.planner_preload_mb * (1 << 20))
    def execute(plan, target_ms):
        """Build the planned workload, run it streamed, return one result row."""
        streamed_layers = int(((plan["keep"] > 0) & (plan["preload"] == 0)).any(axis=1).sum())
        work = W.make_planned(plan["keep"], plan["bits"], plan["preload"], batch=B, seq=L, workers=workers,
                              ring_slots=max(2, min(ring, streamed_layers)))
        kept_bits = plan["bits"][plan["keep"] > 0]
        with sti.Session(work, compute_stream=stream.cuda_stream) as sess:
            x = device_act(torch, work)
            y = torch.empty_like(x)
            ms = forward_ms(sess, work, x, y, args.steps)
            sti.sti_plan_set_profiling(sess.plan, 1)
            stall, copy = [], []
            with torch.cuda.stream(stream):
                for _ in range(5):
                    flush.zero_()
                    sti.sti_model_forward(sess.plan, x.data_ptr(), y.data_ptr(), B, L)
                    st = sti.sti_get_stats(sess.plan)
                    stall.append(sum(st.stall_us[:st.n_layers]))
                    copy.append(sum(st.copy_us[:st.n_layers]))
            sti.sti_plan_set_profiling(sess.plan, 0)
            mem = sti.sti_plan_memory(sess.plan)
        stall_us, copy_us = float(np.median(stall)), float(np.median(copy))
        return {
            "target_ms": target_ms, "n": plan["n"], "m": plan["m"], "pass1_bits": plan["pass1_bits"],
            "valid": plan["valid"], "bits_hist": {int(b): int((kept_bits == b).sum()) for b in np.unique(kept_bits)},
            "mean_bits": float(kept_bits.astype(np.float64).mean()),
            "preloaded_shards": int(plan["preload"].sum()), "preload_bytes_used": mem["preload_bytes"],
            "predicted_ms": plan["n"] * t_comp_us[plan["m"]] * 1e-3, "measured_ms": ms,
            "meets_target": ms <= target_ms, "streamed_bytes": work.packed_bytes() - mem["preload_bytes"],
            "h2d_copy_ms": copy_us * 1e-3, "stall_ms": stall_us * 1e-3,
            "hidden_frac": 1.0 - stall_us / copy_us if copy_us > 0 else None,
            "min_aib_us": float(plan["aib_us"][:plan["n"]].min())}

    rows = []
    targets = [float(t) for t in args.planner_targets_ms.split(",")]
    for target_ms in targets:
        plan = sti.sti_plan_auto(target_ms * 1e3, N, M, t_comp_us, t_io_us, shard_bytes, importance, preload_bytes)
        rows.append(execute(plan, target_ms))

    # back-to-back executions (Section 3.2): the buffer grows between runs, the shards already loaded stay
    # cached bottom-up ON THE DEVICE (sti_plan_retain / sti_shard_adopt: one context, the next plan takes over what
    # the previous one holds and uploads only the rest), and the next plan spends the freed IO time on higher
    # versions of the other shards
    series = []
    target_ms = targets[-1]
    buffers = [int(float(v) * (1 << 20)) for v in args.planner_series_mb.split(",")]
    plan, prev, ctx = None, None, 0
    plans_alive = []
    try:
        for step, buf in enumerate(buffers):
            cached = None
            if plan is not None:
                cached, _ = sti.sti_preload_after_run(plan["keep"], plan["bits"], shard_bytes, buf)
            plan = sti.sti_plan_auto(target_ms * 1e3, N, M, t_comp_us, t_io_us, shard_bytes, importance, buf, cached)
            streamed_layers = int(((plan["keep"] > 0) & (plan["preload"] == 0)).any(axis=1).sum())
            work = W.make_planned(plan["keep"], plan["bits"], plan["preload"], batch=B, seq=L, workers=workers,
                                  ring_slots=max(2, min(ring, streamed_layers)))
            sh = work.shape
            desc = sti.StiModelDesc(n_layers=sh.n_layers, hidden=sh.hidden, n_heads=sh.n_heads, head_dim=sh.head_dim,
                                    ffn=sh.ffn, n_ffn_slices=sh.n_ffn_slices, max_batch=B, max_seq=L,
                                    act_dtype=sti.STI_BF16 if work.act_dtype == "bf16" else sti.STI_F32,
                                    ln_eps=work.ln_eps)
            if not ctx:
                ctx = sti.sti_ctx_create(desc, 0, stream.cuda_stream)
                for l, p in enumerate(work.dense):
                    sti.sti_ctx_set_layer_params(ctx, l, p["bq"], p["bk"], p["bv"], p["bo"], p["b1"], p["b2"],
                                                 p["ln1_g"], p["ln1_b"], p["ln2_g"], p["ln2_b"])
            attn = [(u.keep, u.bits, u.resident) for layer in work.attn_plan for u in layer]
            ffn = [(u.keep, u.bits, u.resident) for layer in work.ffn_plan for u in layer]
            handle = sti.sti_plan_create(ctx, attn, ffn, work.ring_slots)
            plans_alive.append(handle)
            for (l, kind, idx), b in work.blobs.items():
                if cached is not None and cached[l][idx] != 0:
                    sti.sti_shard_adopt(handle, prev, l, kind, idx)
                else:
                    sti.sti_shard_upload(handle, l, kind, idx, b.bits, b.codes, b.centroids, b.outlier_off, b.outlier_val)
            sti.sti_plan_finalize(handle)
            fill = sti.sti_plan_fill_stats(handle)
            if prev:                                            # the previous plan has handed its shards over
                sti.sti_plan_destroy(prev)
                plans_alive.remove(prev)
            x = device_act(torch, work)
            y = torch.empty_like(x)
            retained = 0
            if step + 1 < len(buffers):                         # what the next execution will find cached stays on the device
                keep_next, _ = sti.sti_preload_after_run(plan["keep"], plan["bits"], shard_bytes, buffers[step + 1])
                mask = (keep_next != 0).astype(np.uint8)
                retained = sti.sti_plan_retain(handle, mask, mask)
            ms = []
            with torch.cuda.stream(stream):
                for i in range(3 + args.steps):
                    flush.zero_()
                    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                    e0.record(stream)
                    sti.sti_model_forward(handle, x.data_ptr(), y.data_ptr(), B, L)
                    e1.record(stream)
                    stream.synchronize()
                    if i >= 3:
                        ms.append(e0.elapsed_time(e1))
            sti.sti_plan_set_profiling(handle, 1)
            stall = []
            with torch.cuda.stream(stream):
                for _ in range(5):
                    flush.zero_()
                    sti.sti_model_forward(handle, x.data_ptr(), y.data_ptr(), B, L)
                    st = sti.sti_get_stats(handle)
                    stall.append(sum(st.stall_us[:st.n_layers]))
            sti.sti_plan_set_profiling(handle, 0)
            sti.sti_sync(ctx)
            kept_bits = plan["bits"][plan["keep"] > 0]
            series.append({"buffer_mb": buf / (1 << 20), "n": plan["n"], "m": plan["m"], "pass1_bits": plan["pass1_bits"],
                           "bits_hist": {int(b): int((kept_bits == b).sum()) for b in np.unique(kept_bits)},
                           "mean_bits": float(kept_bits.astype(np.float64).mean()),
                           "preloaded_shards": int(plan["preload"].sum()),
                           "cached_shards_taken_over": 0 if cached is None else int((cached != 0).sum()),
                           "uploaded_bytes": fill["uploaded_bytes"], "adopted_bytes": fill["adopted_bytes"],
                           "retained_bytes_for_next": int(retained),
                           "measured_ms": float(np.median(ms)), "meets_target": bool(np.median(ms) <= target_ms),
                           "stall_ms": float(np.median(stall)) * 1e-3})
            prev = handle
    finally:
        for h in plans_alive:
            sti.sti_plan_destroy(h)
        if ctx:
            sti.sti_ctx_destroy(ctx)

    print(json.dumps({"planner": "two-stage planner on profiled device tables, BERT-large 24x16 store",
                      "batch": B, "seq": L, "preload_budget_bytes": preload_bytes, "h2d_GBps": h2d_gbps,
                      "shard_bytes": shard_bytes, "t_io_us": t_io_us, "t_comp_us": t_comp_us[1:],
                      "pipeline_us_per_layer": pipe_us, "t_comp16_us_resident_2bit": measured[-1],
                      "t_comp16_us_resident_6bit": t_comp16_6bit,
                      "ring_slots": ring, "rows": rows, "back_to_back": series}))


def planner_point(args, target_ms):
    """One planner-made plan, end to end, for the default bench line: profile the device on three submodel widths,
    let sti_plan_auto choose the submodel, the bitwidths and the preload prefix for `target_ms`, execute it streamed
    and report what the pipeline hid (Section 5)."""
    pf = planner_profile(args, widths=(4, 8, 16))
    W, sti, torch, stream, flush, forward_ms = pf["W"], pf["sti"], pf["torch"], pf["stream"], pf["flush"], pf["forward_ms"]
    B, L, N, M = pf["B"], pf["L"], pf["N"], pf["M"]
    importance = np.random.default_rng(np.random.SeedSequence([0, 77])).uniform(0, 1, (N, M)).astype(np.float32)
    preload_bytes = int(args.planner_preload_mb * (1 << 20))
    plan = sti.sti_plan_auto(target_ms * 1e3, N, M, pf["t_comp_us"], pf["t_io_us"], pf["shard_bytes"], importance,
                             preload_bytes)
    streamed_layers = int(((plan["keep"] > 0) & (plan["preload"] == 0)).any(axis=1).sum())
    work = W.make_planned(plan["keep"], plan["bits"], plan["preload"], batch=B, seq=L, workers=pf["workers"],
                          ring_slots=max(2, min(pf["ring"], streamed_layers)))
    kept_bits = plan["bits"][plan["keep"] > 0]
    with sti.Session(work, compute_stream=stream.cuda_stream) as sess:
        x = device_act(torch, work)
        y = torch.empty_like(x)
        ms = forward_ms(sess, work, x, y, 10)
        sti.sti_plan_set_profiling(sess.plan, 1)
        stall, copy = [], []
        with torch.cuda.stream(stream):
            for _ in range(5):
                flush.zero_()
                sti.sti_model_forward(sess.plan, x.data_ptr(), y.data_ptr(), B, L)
                st = sti.sti_get_stats(sess.plan)
                stall.append(sum(st.stall_us[:st.n_layers]))
                copy.append(sum(st.copy_us[:st.n_layers]))
        sti.sti_plan_set_profiling(sess.plan, 0)
    stall_us, copy_us = float(np.median(stall)), float(np.median(copy))
    return {"workload": "two-stage planner (Section 5) on this device's measured T_comp / T_io, BERT-large 24x16 store, "
                        f"batch {B}, seq {L}, {args.planner_preload_mb:g} MiB preload buffer, seeded uniform importance",
            "target_ms": target_ms, "n": plan["n"], "m": plan["m"], "pass1_bits": plan["pass1_bits"],
            "mean_bits": float(kept_bits.astype(np.float64).mean()), "preloaded_shards": int(plan["preload"].sum()),
            "predicted_ms": plan["n"] * pf["t_comp_us"][plan["m"]] * 1e-3, "measured_ms": ms,
            "meets_target": bool(ms <= target_ms), "h2d_copy_ms": copy_us * 1e-3, "stall_ms": stall_us * 1e-3,
            "hidden_frac": 1.0 - stall_us / copy_us if copy_us > 0 else None, "h2d_GBps": pf["h2d_gbps"]}


def decode_rate_point(sti, torch, sess, work, stream, flush, peaks, token_counts=(8, 32, 128), reps=7):
    """Steady-state rate of the fused decode: ONE launch over the FFN1 tiles of all layers (sti_decode_rate_probe), timed
    with events, at few tokens where the decode is all there is to do.  Packed bytes per second against the HBM roof."""
    d, n_layers, ffn = work.shape.hidden, work.shape.n_layers, work.shape.ffn
    out = {"what": "one launch of the dequant-GEMM over every layer's FFN1 tiles (weights resident, cold L2)"}
    for T in token_counts:
        x = torch.randn(T, d, device="cuda").to(torch.bfloat16)
        y = torch.empty(T, n_layers * ffn, dtype=torch.bfloat16, device="cuda")
        ms = []
        packed = tiles = 0
        with torch.cuda.stream(stream):
            for i in range(reps + 2):
                flush.zero_()
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                packed, tiles = sti.sti_decode_rate_probe(sess.plan, x.data_ptr(), T, y.data_ptr(), y.numel() * 2)
                e1.record(stream)
                stream.synchronize()
                if i >= 2:
                    ms.append(e0.elapsed_time(e1))
        t = float(np.median(ms)) * 1e-3
        out[f"tokens_{T}"] = {"ms": t * 1e3, "tiles": tiles, "packed_bytes": packed, "packed_GBps": packed / t / 1e9,
                              "frac_of_hbm": packed / t / 1e9 / float(peaks["hbm_gbs"]),
                              "weights_per_s": n_layers * ffn * d / t}
    return out


def model_point(sti, torch, work, stream, flush, peaks, label, steps=12, warm=4):
    """A model workload resident and streamed: forward ms (median, cold L2), the dequant-GEMMs' stamped time and
    TFLOP/s under graph replay, and how much of the host-to-device copy time the pipeline hid."""
    n_layers = work.shape.n_layers
    B, L = work.batch, work.seq
    x = device_act(torch, work)
    y = torch.empty_like(x)
    out = {"workload": label, "tokens": B * L, "n_layers": n_layers, "packed_bytes": work.packed_bytes()}

    def median_ms(sess):
        ms = []
        with torch.cuda.stream(stream):
            for i in range(warm + steps):
                flush.zero_()
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                sti.sti_model_forward(sess.plan, x.data_ptr(), y.data_ptr(), B, L)
                e1.record(stream)
                stream.synchronize()
                if i >= warm:
                    ms.append(e0.elapsed_time(e1))
        sti.sti_sync(sess.ctx)
        return float(np.median(ms))

    with sti.Session(with_residency(work, n_layers), compute_stream=stream.cuda_stream) as sess:
        out["ms_resident"] = median_ms(sess)
        per, count, total = stamped_forwards(sti, torch, sess, stream, flush, x, y, B, L, n_layers, reps=5)
        gemm_s = float(sum(per[k] for k in GEMM_KERNELS)) * 1e-6
        out.update({"gemm_ms": gemm_s * 1e3, "gemm_TFLOPs": gemm_flops(work) / gemm_s / 1e12,
                    "gemm_frac_of_tensor_peak": gemm_flops(work) / gemm_s / 1e12 / peaks["bf16_tflops_sustained"],
                    "forward_TFLOPs": (gemm_flops(work) + attn_flops(work)) / (out["ms_resident"] * 1e-3) / 1e12,
                    "packed_GBps_resident": work.packed_bytes() / (out["ms_resident"] * 1e-3) / 1e9,
                    "kernel_us_per_layer": {KERNEL_NAMES[k]: float(per[k] / n_layers) for k in range(1, 8)}})
    with sti.Session(work, compute_stream=stream.cuda_stream) as sess:
        out["ms_streamed"] = median_ms(sess)
        sti.sti_plan_set_profiling(sess.plan, 1)
        with torch.cuda.stream(stream):
            for _ in range(3):
                flush.zero_()
                sti.sti_model_forward(sess.plan, x.data_ptr(), y.data_ptr(), B, L)
                st = sti.sti_get_stats(sess.plan)
        sti.sti_plan_set_profiling(sess.plan, 0)
        copy_ms = sum(st.copy_us[:st.n_layers]) * 1e-3
        out.update({"h2d_copy_ms": copy_ms, "stall_ms": sum(st.stall_us[:st.n_layers]) * 1e-3,
                    "streamed_bytes": int(sum(st.streamed_bytes[:st.n_layers])),
                    "hidden_frac": 1.0 - max(0.0, out["ms_streamed"] - out["ms_resident"]) / copy_ms if copy_ms > 0 else None,
                    "hidden_frac_cap": min(1.0, out["ms_resident"] / copy_ms) if copy_ms > 0 else None,
                    "streamed_over_resident": out["ms_streamed"] / out["ms_resident"]})
    return out


def run_baselines(args):
    """Section 7.1's comparison systems as plans of this library, next to the two-stage planner, for the same
    target latencies on the same profiled device tables (latency only; accuracy needs trained weights):
      Load&Exec       32-bit shards, everything loaded before layer 0 starts (IO + compute add up)
      StdPL-X         uniform X bits, layerwise pipeline, nothing preloaded
      PreloadModel-X  uniform X bits, the whole submodel resident (no IO at run time)
      STI             sti_plan_auto: per-shard bitwidths, preload prefix, layerwise pipeline
    Each baseline picks the submodel with Section 5.3's rule (most shards, then deepest) under its own
    delay model, the plan is executed, and measured latency, fidelity (bits) and memory are reported."""
    pf = planner_profile(args)
    W, sti, torch, stream, flush, forward_ms = pf["W"], pf["sti"], pf["torch"], pf["stream"], pf["flush"], pf["forward_ms"]
    B, L, N, M, workers = pf["B"], pf["L"], pf["N"], pf["M"], pf["workers"]
    versions, shard_bytes, t_io_us, t_comp_us = pf["versions"], pf["shard_bytes"], pf["t_io_us"], pf["t_comp_us"]
    importance = np.random.default_rng(np.random.SeedSequence([0, 77])).uniform(0, 1, (N, M)).astype(np.float32)
    preload_bytes = int(args.planner_preload_mb * (1 << 20))
    X = args.baseline_bits
    vi = {k: i for i, k in enumerate(versions)}

    def pick(delay_us, target_us):
        best = None
        for n in range(1, N + 1):
            for m in range(1, M + 1):
                if delay_us(n, m) <= target_us and (best is None or n * m > best[0] * best[1] or
                                                    (n * m == best[0] * best[1] and n > best[0])):
                    best = (n, m)
        return best

    def pipeline_us(n, m, bits):
        """Layerwise pipeline with nothing preloaded: layer k starts when its shards and layer k-1 are done."""
        io_done = comp_done = 0.0
        for _ in range(n):
            io_done += m * t_io_us[vi[bits]]
            comp_done = max(comp_done, io_done) + t_comp_us[m]
        return comp_done

    def grids(n, m, bits, preload):
        keep = np.zeros((N, M), np.uint8)
        rank = np.argsort(-importance, axis=1, kind="stable")
        for l in range(n):
            keep[l, rank[l, :m]] = 1                     # the m most important shards of the layer
        return keep, keep * bits, keep * (1 if preload else 0)

    def execute(name, keep, bits, preload, target_ms, predicted_us, overlap=True):
        streamed_layers = int(((keep > 0) & (preload == 0)).any(axis=1).sum())
        work = W.make_planned(keep, bits, preload, batch=B, seq=L, workers=workers, ring_slots=max(2, streamed_layers))
        kept_bits = bits[keep > 0]
        with sti.Session(work, compute_stream=stream.cuda_stream) as sess:
            if not overlap:
                sti.sti_plan_set_overlap(sess.plan, False)
            x = device_act(torch, work)
            y = torch.empty_like(x)
            ms = forward_ms(sess, work, x, y, args.steps)
            mem = sti.sti_plan_memory(sess.plan)
        return {"system": name, "target_ms": target_ms, "n": int(keep.any(axis=1).sum()), "m": int(keep[0].sum()),
                "mean_bits": float(kept_bits.astype(np.float64).mean()),
                "bits_hist": {int(b): int((kept_bits == b).sum()) for b in np.unique(kept_bits)},
                "predicted_ms": predicted_us * 1e-3, "measured_ms": ms, "meets_target": bool(ms <= target_ms * 1.02),
                "device_bytes_resident": mem["preload_bytes"], "device_bytes_ring": mem["ring_bytes"],
                "streamed_bytes": max(0, work.packed_bytes() - mem["preload_bytes"])}

    rows = []
    for target_ms in [float(t) for t in args.planner_targets_ms.split(",")]:
        T = target_ms * 1e3
        # Load&Exec: IO of all 32-bit shards, then compute
        load_exec = lambda n, m: n * m * t_io_us[vi[32]] + n * t_comp_us[m]
        nm = pick(load_exec, T)
        if nm:
            rows.append(execute("Load&Exec", *grids(nm[0], nm[1], 32, False), target_ms, load_exec(*nm), overlap=False))
        else:
            rows.append({"system": "Load&Exec", "target_ms": target_ms, "n": 0, "m": 0, "note": "no submodel fits"})
        nm = pick(lambda n, m: pipeline_us(n, m, X), T)
        if nm:
            rows.append(execute(f"StdPL-{X}", *grids(nm[0], nm[1], X, False), target_ms, pipeline_us(nm[0], nm[1], X)))
        else:
            rows.append({"system": f"StdPL-{X}", "target_ms": target_ms, "n": 0, "m": 0, "note": "no submodel fits"})
        nm = pick(lambda n, m: n * t_comp_us[m], T)
        rows.append(execute(f"PreloadModel-{X}", *grids(nm[0], nm[1], X, True), target_ms, nm[0] * t_comp_us[nm[1]]))
        plan = sti.sti_plan_auto(T, N, M, t_comp_us, t_io_us, shard_bytes, importance, preload_bytes)
        rows.append(execute("STI", plan["keep"], plan["bits"], plan["preload"], target_ms,
                            plan["n"] * t_comp_us[plan["m"]]))
    print(json.dumps({"baselines": "Section 7.1 systems as plans, BERT-large 24x16 store", "batch": B, "seq": L,
                      "X": X, "preload_budget_bytes": preload_bytes, "h2d_GBps": pf["h2d_gbps"],
                      "t_io_us": t_io_us, "t_comp_us": t_comp_us[1:], "rows": rows}))


def shape_layers_default():
    """The quantizer's default workload is the whole model: every launch then holds more units than the GPU has SMs."""
    import workloads as W
    return W.BERT_LARGE.n_layers


def run_quantize(args):
    """Section 6 on the device: every shard unit of `--layers` BERT-large layers (default: all 24; 16 attention units of 262,144
    weights and 16 FFN units of 524,288 weights per layer) quantized at `--baseline-bits` bits by
    sti_quantize_units, timed with CUDA events, next to the CPU oracle on a sample of the same units."""
    import workloads as W
    from workloads.shards import ATTN, FFN, make_unit_weights
    from oracle import sti_quantizer_oracle as Q
    n_layers = args.layers or shape_layers_default()
    bits = args.baseline_bits
    shape = W.BERT_LARGE
    groups = {}
    for kind, name in ((ATTN, "attn"), (FFN, "ffn")):
        groups[name] = np.stack([np.concatenate([m.reshape(-1) for m in make_unit_weights(shape, 0, l, kind, i)])
                                 for l in range(n_layers) for i in range(shape.n_heads)])
    t0 = time.perf_counter()
    sample = [groups["attn"][0], groups["ffn"][0]]
    for u in sample:
        Q.quantize_unit(u, bits)
    cpu_s = time.perf_counter() - t0
    cpu_weights = sum(u.size for u in sample)
    import torch
    import paper_2207_05022_b200 as sti
    from paper_2207_05022_b200 import build
    build.build_library()
    peaks, peak_src = load_peaks()
    stream = torch.cuda.current_stream()
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    rows, total_ms, total_weights, total_bytes = [], 0.0, 0, 0
    for method, name, units in [(m, nm, u) for m in ("select", "sort") for nm, u in groups.items()]:
        n_units, n = units.shape
        w = torch.from_numpy(units).cuda()
        codes = torch.zeros((n_units, n * bits // 32), dtype=torch.int32, device="cuda")
        cents = torch.zeros((n_units, 1 << bits), dtype=torch.float32, device="cuda")
        off = torch.zeros((n_units, 4096), dtype=torch.int32, device="cuda")
        val = torch.zeros((n_units, 4096), dtype=torch.float32, device="cuda")
        cnt = torch.zeros(n_units, dtype=torch.int32, device="cuda")
        ws_bytes = sti.sti_quantize_workspace_bytes(n_units, n)
        ws = torch.empty(ws_bytes, dtype=torch.uint8, device="cuda")
        ms = []
        for i in range(args.warmup + args.steps):
            flush.zero_()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            sti.sti_quantize_units_by(w.data_ptr(), n_units, n, bits, codes.data_ptr(), cents.data_ptr(), off.data_ptr(),
                                      val.data_ptr(), 4096, cnt.data_ptr(), ws.data_ptr(), ws_bytes,
                                      sti.STI_QUANTIZE_SELECT if method == "select" else sti.STI_QUANTIZE_SORT,
                                      stream=stream.cuda_stream)
            e1.record(stream)
            stream.synchronize()
            if i >= args.warmup:
                ms.append(e0.elapsed_time(e1))
        med = float(np.median(ms))
        algo = n_units * (n * 4 + n * bits // 8 + (4 << bits))            # fp32 in, index stream + table out
        rows.append({"method": method, "units": name, "n_units": n_units, "weights_per_unit": n, "ms": med,
                     "Mweights_per_s": n_units * n / med / 1e3, "algorithmic_GBps": algo / med / 1e6,
                     "frac_of_hbm_peak": algo / med / 1e6 / peaks["hbm_gbs"], "workspace_bytes": ws_bytes,
                     "outliers_mean": float(cnt.float().mean().item())})
        if method == "select":                                            # the library's default is the headline
            total_ms += med; total_weights += n_units * n; total_bytes += algo
        del w, codes, cents, off, val, cnt, ws
    print(json.dumps({"quantize": f"Section 6 quantizer, {n_layers} BERT-large layers, {bits} bits", "rows": rows,
                      "total_ms": total_ms, "Mweights_per_s": total_weights / total_ms / 1e3,
                      "roofline": {"bound": "hbm", "achieved": total_bytes / total_ms / 1e6, "peak": peaks["hbm_gbs"],
                                   "unit": "GB/s", "frac": total_bytes / total_ms / 1e6 / peaks["hbm_gbs"],
                                   "traffic": None, "peak_source": f"hbm_gbs, {peak_src}",
                                   "note": "totals are the selecting method's (the default); a cluster of CTAs per unit, two passes "
                                           "over the unit's fp32 weights"},
                      "cpu_baseline": {"value": cpu_weights / cpu_s / 1e6, "unit": "Mweights/s", "cores": blas_threads(),
                                       "kind": "oracle", "sample": "one attention unit and one FFN unit of layer 0"}}))


GEMM_KERNELS = (1, 3, 5, 6)          # QKV, O projection, FFN1, FFN2 in the per-layer stamp records
KERNEL_NAMES = ("cast", "qkv", "attention", "o_proj", "layernorm1", "ffn1", "ffn2", "layernorm2")


def stamp_intervals(stamps):
    """Per-kernel share of one forward from the kernels' own device-timer stamps (profiling level 3, graph replay).

    Kernels overlap (each is launched before its predecessor ends and decodes its weights meanwhile), so a kernel's
    time is taken as the interval from the previous kernel's last-CTA end to its own: the intervals of a forward add
    up to the forward.  Returns (us per kernel slot summed over layers [8], launches per slot [8], total us)."""
    n_layers = stamps.shape[0]
    per = np.zeros(8)
    count = np.zeros(8, dtype=np.int64)
    prev_end = None
    first = None
    for l in range(n_layers):
        for k in range(8):
            end = int(stamps[l, k, 2])
            if end == 0:
                continue                                   # this kernel did not run
            if prev_end is None:
                prev_end = first = int(stamps[l, k, 0])    # the forward's first kernel: from its first CTA's start
            per[k] += (end - prev_end) * 1e-3
            count[k] += 1
            prev_end = end
    total = (prev_end - first) * 1e-3 if prev_end is not None else 0.0
    return per, count, total


def stamped_forwards(sti, torch, sess, stream, flush, x, y, B, L, n_layers, reps, warm=2):
    """Runs `reps` graph-replayed forwards with kernel stamps on (cold L2 each) and returns the mean per-kernel
    interval sums, the launches per kernel slot and the mean stamped total, all per forward."""
    sti.sti_plan_set_profiling(sess.plan, 3)
    per_acc, total_acc, count = np.zeros(8), 0.0, np.zeros(8, dtype=np.int64)
    with torch.cuda.stream(stream):
        for i in range(warm + reps):
            flush.zero_()
            sti.sti_model_forward(sess.plan, x.data_ptr(), y.data_ptr(), B, L)
            stream.synchronize()
            if i >= warm:
                per, count, total = stamp_intervals(sti.sti_get_kernel_stamps(sess.plan, n_layers))
                per_acc += per
                total_acc += total
    sti.sti_plan_set_profiling(sess.plan, 0)
    return per_acc / reps, count, total_acc / reps


def plain_h2d_gbps(torch, stream, mb=64, reps=8):
    """Pinned host -> device cudaMemcpyAsync rate of the box, measured alone (the denominator of the streamed arm)."""
    src = torch.empty(mb << 20, dtype=torch.uint8).pin_memory()
    dst = torch.empty(mb << 20, dtype=torch.uint8, device="cuda")
    rates = []
    with torch.cuda.stream(stream):
        for i in range(reps + 2):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            dst.copy_(src, non_blocking=True)
            e1.record(stream)
            stream.synchronize()
            if i >= 2:
                rates.append(src.numel() / (e0.elapsed_time(e1) * 1e-3) / 1e9)
    return float(np.median(rates))


def oracle_single_thread(work, layers):
    """The oracle on one host thread (BLAS pool limited to 1) over `layers`; returns seconds."""
    try:
        from threadpoolctl import threadpool_limits
    except Exception:
        return None
    with threadpool_limits(limits=1):
        return oracle_forward_timed(work, layers)


def spawn_ranks(n, argv, extra_env=None, port=None):
    """Starts `n` copies of the command `argv`, one per GPU of this node, with the rendezvous variables torchrun would
    set (RANK, LOCAL_RANK, WORLD_SIZE, MASTER_ADDR=127.0.0.1, MASTER_PORT); rank 0 inherits stdout, the others'
    output goes to stderr.  Returns the largest exit code."""
    port = port or (29500 + os.getpid() % 2000)
    procs = []
    for r in range(n):
        env = dict(os.environ)
        env.update({"RANK": str(r), "LOCAL_RANK": str(r), "WORLD_SIZE": str(n), "LOCAL_WORLD_SIZE": str(n),
                    "MASTER_ADDR": "127.0.0.1", "MASTER_PORT": str(port)})
        env.setdefault("NCCL_DEBUG", "INFO")               # the communicator's transport choices stay visible
        if extra_env:
            env.update(extra_env)
        procs.append(subprocess.Popen(list(argv), env=env, stdout=None if r == 0 else sys.stderr))
    codes = [p.wait() for p in procs]
    return max(codes)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--layers", type=int, default=0, help="shorten the stack (profiler captures only)")
    ap.add_argument("--no-extras", action="store_true", help="skip the cpu baseline and single-layer extras")
    ap.add_argument("--sweep", action="store_true", help="configuration 5 sweep instead of the headline workload")
    ap.add_argument("--sweep-batches", default="1,8,32,64")
    ap.add_argument("--sweep-seqs", default="128,512")
    ap.add_argument("--planner", action="store_true", help="profile, plan with sti_plan_auto and run the plans")
    ap.add_argument("--planner-batch", type=int, default=1)
    ap.add_argument("--planner-seq", type=int, default=256)
    ap.add_argument("--planner-targets-ms", default="0.4,0.8,1.6,3.2")
    ap.add_argument("--planner-preload-mb", type=float, default=8.0)
    ap.add_argument("--planner-series-mb", default="8,32,64",
                    help="preload buffer sizes of consecutive back-to-back executions at the last target")
    ap.add_argument("--baselines", action="store_true",
                    help="Load&Exec / StdPL-X / PreloadModel-X / planner comparison on the profiled device")
    ap.add_argument("--quantize", action="store_true", help="time the device quantizer (Section 6) on BERT-large units")
    ap.add_argument("--baseline-bits", type=int, default=6, choices=[2, 3, 4, 5, 6])
    ap.add_argument("--planner-ring", type=int, default=24,
                    help="most streamed-layer buffers on the device (the IO budgets assume loading runs ahead freely)")
    args = ap.parse_args()
    if args.impl == "reference":
        run_reference(args)
        return
    if args.sweep:
        args.steps = min(args.steps, 10)
        run_sweep(args)
        return
    if args.planner:
        args.steps = min(args.steps, 20)
        run_planner(args)
        return
    if args.quantize:
        args.steps = min(args.steps, 10)
        run_quantize(args)
        return
    if args.baselines:
        args.steps = min(args.steps, 20)
        run_baselines(args)
        return
    args.warmup = max(args.warmup, 3)
    if args.gpus > 1 and "WORLD_SIZE" not in os.environ:
        # launched plainly with --gpus N: start the N replicas ourselves (the path has no exchange step: one
        # independent replica per GPU; NCCL only carries the barrier and the max-over-ranks reduction)
        raise SystemExit(spawn_ranks(args.gpus, [sys.executable, os.path.abspath(__file__)] + sys.argv[1:]))

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))

    # inputs first: the quantizer pool is spawned before the first CUDA call
    import workloads as W
    workers = min(8, os.cpu_count() or 1)
    work_str = W.make_config(4, n_layers=args.layers or None, workers=workers)
    work_res = with_residency(work_str, work_str.shape.n_layers)
    packed = work_str.packed_bytes()

    cpu_baseline = None
    if rank == 0 and world == 1 and not args.no_extras:
        # the oracle as it stands on the whole model, repeated until about ten seconds of CPU work have been timed
        n_sample = work_str.shape.n_layers
        secs, reps = 0.0, 0
        while reps < 4 and secs < 10.0:
            secs += oracle_forward_timed(work_str, list(range(n_sample)))
            reps += 1
        cpu_baseline = {"value": work_str.packed_bytes(range(n_sample)) * reps / secs / 1e9, "unit": UNIT,
                        "cores": blas_threads(), "kind": "oracle", "seconds": secs,
                        "sample": f"all {n_sample} layers, decode + fp64 forward, {reps} times"}
        one = list(range(min(2, n_sample)))
        secs1 = oracle_single_thread(work_str, one)
        if secs1:
            cpu_baseline["single_thread"] = {"value": work_str.packed_bytes(one) / secs1 / 1e9, "unit": UNIT, "cores": 1,
                                             "seconds": secs1, "sample": f"layers 0-{one[-1]}, once"}

    import torch
    import torch.distributed as dist
    import paper_2207_05022_b200 as sti
    from paper_2207_05022_b200 import build
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device: the library has no CPU execution path")
    build.build_library()
    sti.load_library()
    torch.cuda.set_device(local_rank)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local_rank))

    def barrier():
        torch.cuda.synchronize()
        if world > 1:
            dist.barrier()

    peaks, peak_src = load_peaks()
    for k, v in FALLBACK_PEAKS.items():
        peaks.setdefault(k, v)
    stream = torch.cuda.Stream()
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    x_dev = torch.from_numpy(work_str.x_dev).cuda()
    y_dev = torch.empty_like(x_dev)
    x_host = torch.from_numpy(work_str.x_dev).pin_memory()
    y_host = torch.empty_like(x_host).pin_memory()
    B, L = work_str.batch, work_str.seq
    K, Wm = args.steps, args.warmup

    s_res = sti.Session(work_res, device=local_rank, compute_stream=stream.cuda_stream)
    s_str = sti.Session(work_str, device=local_rank, compute_stream=stream.cuda_stream)
    sampler = ClockSampler(local_rank)

    def timed(fn, cold=True):
        """W warm-up steps, then exactly K timed ones; returns (job time of the K steps in ms, max over ranks;
        this rank's per-step times)."""
        with torch.cuda.stream(stream):
            for _ in range(Wm):
                if cold:
                    flush.zero_()
                fn()
            barrier()
            ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(K)]
            for e0, e1 in ev:
                if cold:
                    flush.zero_()                 # cold L2 for every step (outside the timed interval)
                e0.record(stream)
                fn()
                e1.record(stream)
            barrier()
        steps = [e0.elapsed_time(e1) for e0, e1 in ev]
        return max_over_ranks(sum(steps), world), steps

    sampler.start()
    launches0 = sti.sti_ctx_launch_count(s_res.ctx)
    ms_res, steps_res = timed(lambda: sti.sti_model_forward(s_res.plan, x_dev.data_ptr(), y_dev.data_ptr(), B, L))
    launches = sti.sti_ctx_launch_count(s_res.ctx) - launches0
    sti.sti_sync(s_res.ctx)
    ms_e2e, steps_e2e = timed(lambda: sti.sti_model_forward_host(s_str.plan, x_host.data_ptr(), y_host.data_ptr(), B, L))
    sti.sti_sync(s_str.ctx)
    ms_str_dev, _ = timed(lambda: sti.sti_model_forward(s_str.plan, x_dev.data_ptr(), y_dev.data_ptr(), B, L))
    sti.sti_sync(s_str.ctx)
    clocks = sampler.stop()
    # the same forward with whatever the previous step left in L2 (packed weights are 136 MB, L2 126 MB)
    ms_warm, _ = timed(lambda: sti.sti_model_forward(s_res.plan, x_dev.data_ptr(), y_dev.data_ptr(), B, L), cold=False)
    sti.sti_sync(s_res.ctx)

    # the dominant kernel's time in the SAME execution mode as the timed value: device-timer stamps written by the
    # kernels themselves under graph replay
    n_layers = work_str.shape.n_layers
    per_kernel_us, kernel_count, stamped_total_us = stamped_forwards(sti, torch, s_res, stream, flush, x_dev, y_dev, B, L,
                                                                      n_layers, reps=min(K, 10))
    gemm_us = float(sum(per_kernel_us[k] for k in GEMM_KERNELS))         # per forward
    gemm_launches = int(sum(kernel_count[k] for k in GEMM_KERNELS))      # per forward
    attn_us, ln_us = float(per_kernel_us[2]), float(per_kernel_us[4] + per_kernel_us[7])
    # streamed run: copy durations and stalls
    sti.sti_plan_set_profiling(s_str.plan, 1)
    copy_us = stall_us = 0.0
    streamed_bytes = 0
    with torch.cuda.stream(stream):
        for i in range(3):
            flush.zero_()
            sti.sti_model_forward(s_str.plan, x_dev.data_ptr(), y_dev.data_ptr(), B, L)
            st = sti.sti_get_stats(s_str.plan)
            copy_us, stall_us = sum(st.copy_us[:st.n_layers]), sum(st.stall_us[:st.n_layers])
            streamed_bytes = sum(st.streamed_bytes[:st.n_layers])
    sti.sti_plan_set_profiling(s_str.plan, 0)
    mem = sti.sti_plan_memory(s_str.plan)
    h2d_plain = plain_h2d_gbps(torch, stream) if rank == 0 else None

    decode_rate = decode_rate_point(sti, torch, s_res, work_str, stream, flush, peaks) if rank == 0 else None

    s_res.close()
    s_str.close()
    extras = {}
    if rank == 0 and world == 1 and not args.no_extras:
        # configurations 1 and 2 (single BERT-base layers) and the few-token probes of the same layer
        for num in (1, 2):
            extras[f"config{num}_layer"] = time_layer_config(sti, torch, num, peaks)
        for probe_seq in (8, 32):
            extras[f"config1_layer_probe_seq{probe_seq}"] = time_layer_config(sti, torch, 1, peaks, seq=probe_seq)
        # configuration 3: 12-layer BERT-base, layers 0-2 preloaded, the rest streamed, two ring slots
        extras["config3_model"] = model_point(
            sti, torch, W.make_config(3, workers=workers), stream, flush, peaks,
            "12-layer BERT-base, batch 1, seq 128, per-layer random plan (60-100 % kept, 2-6 bits), "
            "layers 0-2 preloaded, layers 3-11 streamed")
        # configuration 5: two points of the sweep on a 4-layer BERT-large stack (bf16 activations, uniform 3 bits,
        # 2-layer preload when streamed); the whole grid is `bench.py --sweep`
        for b5, s5 in ((8, 512), (32, 512)):
            w5 = W.make_config(5, n_layers=4, plan="uniform3", resident=False, batch=b5, seq=s5, workers=workers)
            extras[f"config5_b{b5}_s{s5}_uniform3"] = model_point(
                sti, torch, w5, stream, flush, peaks,
                f"4-layer BERT-large stack, batch {b5}, seq {s5}, uniform 3-bit plan", steps=6, warm=3)
        extras["planner_plan"] = planner_point(args, target_ms=0.8)

    if rank != 0:
        if world > 1:
            dist.destroy_process_group()
        return

    flops_gemm = gemm_flops(work_str)
    gemm_s = gemm_us * 1e-6                          # per forward (stamped under graph replay)
    ach_tflops = flops_gemm / gemm_s / 1e12 if gemm_s > 0 else 0.0
    peak_tf, peak_hbm = float(peaks["bf16_tflops_sustained"]), float(peaks["hbm_gbs"])
    x_bytes = x_host.numel() * x_host.element_size()
    t_res, t_str = ms_res / K, ms_str_dev / K
    t_h2d = copy_us * 1e-3
    hidden = 1.0 - max(0.0, t_str - t_res) / t_h2d if t_h2d > 0 else None
    t_floor_ms = max((packed + 2 * x_bytes) / (peak_hbm * 1e9),
                     (flops_gemm + attn_flops(work_str)) / (peak_tf * 1e12)) * 1e3
    line = {
        "metric": METRIC, "value": aggregate_throughput(packed, world, t_res) / 1e9, "unit": UNIT, "n_gpus": world,
        "steps": K, "warmup": Wm, "ms_per_step": t_res, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "bf16", "data": "synthetic",
        "config": {"workload": WORKLOAD, "n_layers": work_str.shape.n_layers, "batch": B, "seq": L,
                   "packed_bytes": packed, "code_bytes": work_str.code_bytes(), "parallelism": f"replicas x{world}",
                   "l2": "256 MiB memset before every step; packed weights (136 MB) also exceed the 126 MB L2",
                   "value_arm": "all shards resident in device memory",
                   "e2e_arm": "2-layer preload, layers 2.. streamed from pinned host memory"},
        "e2e": {"value": aggregate_throughput(packed, world, ms_e2e / K) / 1e9, "unit": UNIT, "ms_per_step": ms_e2e / K,
                "h2d_bytes_per_step": int(streamed_bytes + x_bytes), "d2h_bytes_per_step": int(x_bytes)},
        "gpu_launches": int(launches),
        "clocks": clocks,
        "roofline": {"kernel": "dqgemm_kernel (fused dequant-GEMM, 4 launches per layer)", "bound": "tensor",
                     "achieved": ach_tflops, "peak": peak_tf, "unit": "TFLOP/s",
                     "frac": ach_tflops / peak_tf if peak_tf else None,
                     "traffic": NCU_DRAM_BYTES_PER_GEMM_LAUNCH if work_str.shape.hidden == 1024 and work_str.seq == 256
                     and work_str.batch == 1 else None,
                     "traffic_note": "dram read+write bytes per launch, mean of a layer's four launches, one ncu "
                                     "capture of this kernel build (cold caches); algorithmic: packed shards + bf16 operands",
                     "peak_source": f"bf16_tflops_sustained, {peak_src}",
                     "flops_per_launch": flops_gemm / gemm_launches if gemm_launches else None,
                     "avg_launch_us": gemm_us / gemm_launches if gemm_launches else None,
                     "launches_per_forward": gemm_launches,
                     "timing": "device-timer stamps written by the kernels during graph-replayed forwards (the timed "
                               "mode); kernels overlap, so a launch's time is the interval from the previous "
                               "kernel's last-CTA end to its own; the intervals of a forward add up to the forward",
                     "hbm_view": {"achieved_GBps": packed / gemm_s / 1e9 if gemm_s > 0 else None, "peak": peak_hbm,
                                  "frac": packed / gemm_s / 1e9 / peak_hbm if gemm_s > 0 else None,
                                  "note": "packed-weight bytes over GEMM time; at 256 tokens the GEMMs are tensor-bound"}},
        "cpu_baseline": cpu_baseline,
        "latency": {"layer_us_mean": t_res * 1e3 / n_layers,
                    "model_ms_resident": t_res, "model_ms_resident_p10": float(np.percentile(steps_res, 10)),
                    "model_ms_resident_p50": float(np.median(steps_res)),
                    "model_ms_resident_p90": float(np.percentile(steps_res, 90)),
                    "model_ms_resident_warm_l2": ms_warm / K,
                    "model_ms_streamed": t_str, "model_ms_e2e_host": ms_e2e / K,
                    "model_ms_e2e_host_p10": float(np.percentile(steps_e2e, 10)),
                    "model_ms_e2e_host_p90": float(np.percentile(steps_e2e, 90)),
                    "roofline_floor_ms": t_floor_ms, "x_of_floor": t_res / t_floor_ms,
                    "stamped_forward_us": stamped_total_us,
                    "gemm_us_per_fwd": gemm_us, "attn_us_per_fwd": attn_us, "ln_us_per_fwd": ln_us,
                    "kernel_us_per_layer": {KERNEL_NAMES[k]: float(per_kernel_us[k] / n_layers) for k in range(1, 8)}},
        "pipeline": {"h2d_copy_ms": t_h2d, "h2d_GBps": streamed_bytes / (t_h2d * 1e-3) / 1e9 if t_h2d > 0 else None,
                     "stall_ms": stall_us * 1e-3, "hidden_frac": hidden,
                     "hidden_frac_cap": min(1.0, t_res / t_h2d) if t_h2d > 0 else None,
                     "pipeline_eff": max(t_h2d, t_res) / t_str if t_str > 0 else None,
                     "h2d_plain_pinned_GBps": h2d_plain,
                     "preload_bytes": mem["preload_bytes"], "pinned_bytes": mem["pinned_bytes"],
                     "ring_bytes": mem["ring_bytes"]},
        "decode_rate": decode_rate,
        "extras": extras,
    }
    print(json.dumps(line))
    if world > 1:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
