"""What this framework is timed on: forwards over dictionary-quantized shards and the quantizer that makes them.

A forward case is a context and a plan as a program keeps them (dense parameters set, shards uploaded, plan finalized)
and one pass over a batch; a quantizer case is a set of fp32 shard units in device memory and the call that turns them
into the upload format.  Shapes are BERT-base and BERT-large; plans keep heads and FFN slices, pick bitwidths and
decide what is resident as the benchmark configurations and the planner do.

The index streams of a forward are uniformly random: clusters hold equally many weights, so that is how a quantized
unit's indexes are distributed.  Their tables are the means of equal-population slices of a normal distribution, and
0.15 % of the weights are outliers, the share the paper reports for trained models.
"""
from __future__ import annotations

import math
import random
from statistics import NormalDist
from types import SimpleNamespace

import numpy as np
import torch

import paper_2207_05022_b200 as sti
from workloads import BERT_BASE, BERT_LARGE, ShardBlob, UnitPlan, unit_weight_count

ATTN, FFN = sti.STI_ATTN, sti.STI_FFN
MODELS = {"base": BERT_BASE, "large": BERT_LARGE}
STD, TAILS = 0.02, 0.0015
# Bitwidths of a plan's units: one version for all, any version, the skew toward 3 bits of a mid budget, and what the
# planner makes of a small one (mostly 2 bits, a few important shards higher, some of them uncompressed).
BIT_MIXES = {"2": ((2,), (1,)), "3": ((3,), (1,)), "4": ((4,), (1,)), "6": ((6,), (1,)),
             "any": ((2, 3, 4, 5, 6), (20, 20, 20, 20, 20)),
             "skew3": ((2, 3, 4, 5, 6), (15, 45, 20, 10, 10)),
             "planned": ((2, 3, 4, 6, 32), (60, 28, 5, 5, 2))}
MAX_TOKENS = 32 * 512


def _forward(name, model, layers, batch, seq, dtype, bits, *, keep=1.0, entry="device", resident=None, slots=2, ragged=False,
             capacity=1, plan=0):
    """entry: "layer" (one layer on device buffers), "device" (the model on device buffers), "host" (the model from and
    to pinned host buffers).  resident: layers in the preload buffer, the others are streamed behind compute.
    capacity: how many times the tokens of this batch the context is sized for.  plan: which units the plan picks."""
    case = {"kind": "forward", "model": model, "layers": layers, "batch": batch, "seq": seq, "dtype": dtype, "bits": bits, "keep": keep,
            "entry": entry, "resident": layers if resident is None else resident, "slots": slots, "ragged": ragged,
            "capacity": capacity, "plan": plan}
    return dict(case, name=name) if name else case


def _quantize(name, units, weights, bits):
    case = {"kind": "quantize", "units": units, "weights": weights, "bits": bits}
    return dict(case, name=name) if name else case


def listed():
    return [
        # one encoder layer called by itself on one short sequence: the smallest call, all latency
        _forward("layer_base_1x128", "base", 1, 1, 128, "f32", "4", entry="layer"),
        # the same call on an elastic layer: two thirds of the heads, mixed bitwidths, bf16 activations
        _forward("layer_base_elastic_1x128", "base", 1, 1, 128, "bf16", "any", keep=0.7, entry="layer"),
        # an interactive query end to end, three layers preloaded, the others streamed from host memory behind compute
        _forward("base_streamed_1x128", "base", 12, 1, 128, "f32", "any", keep=0.8, entry="host", resident=3),
        # the headline configuration with every shard resident
        _forward("large_1x256", "large", 24, 1, 256, "f32", "skew3"),
        # and end to end: two layers preloaded, the others streamed
        _forward("large_streamed_1x256", "large", 24, 1, 256, "f32", "skew3", entry="host", resident=2),
        # a few queries of unequal, odd lengths on a narrowed model, in a context that could take more
        _forward("base_ragged_5x77", "base", 12, 5, 77, "bf16", "skew3", keep=0.75, ragged=True, capacity=2),
        # a small batch through a planner-made submodel (half depth, some shards uncompressed)
        _forward("large_planned_8x128", "large", 12, 8, 128, "bf16", "planned"),
        # a batch of long, unequal sequences
        _forward("large_ragged_8x512", "large", 24, 8, 512, "bf16", "any", ragged=True),
        # throughput: the largest batch
        _forward("large_32x512", "large", 24, 32, 512, "bf16", "3"),
        # making shards: the attention units of one BERT-base layer at one bitwidth
        _quantize("quantize_base_attn_4bit", 12, unit_weight_count(BERT_BASE, ATTN), 4),
        # the FFN units of one BERT-large layer at the highest bitwidth
        _quantize("quantize_large_ffn_6bit", 16, unit_weight_count(BERT_LARGE, FFN), 6),
        # the FFN units of the whole model at the most used one
        _quantize("quantize_large_model_3bit", 384, unit_weight_count(BERT_LARGE, FFN), 3),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    if rng.random() < 0.3:
        if rng.random() < 0.6:
            weights = unit_weight_count(MODELS[rng.choice(("base", "large"))], rng.choice((ATTN, FFN)))
        else:        # other widths: a unit holds a multiple of 128 weights
            weights = 128 * _log_int(rng, 256, 4096)
        return _quantize(None, _log_int(rng, 1, 384), weights, rng.randint(2, 6))
    model = rng.choice(("base", "large"))
    seq = _log_int(rng, 8, 512)
    batch = _log_int(rng, 1, min(64, MAX_TOKENS // seq))
    entry = rng.choice(("layer", "device", "device", "device", "host", "host"))
    layers = 1 if entry == "layer" else _log_int(rng, 2, MODELS[model].n_layers)
    streamed = entry == "host" and rng.random() < 0.7
    tokens = batch * seq
    return _forward(None, model, layers, batch, seq, rng.choice(("f32", "bf16")), rng.choice(sorted(BIT_MIXES)),
                    keep=round(rng.choice((1.0, rng.uniform(0.5, 1.0))), 3), entry=entry,
                    resident=rng.randint(0, min(4, layers)) if streamed else None, slots=rng.randint(2, 4),
                    ragged=batch > 1 and rng.random() < 0.5, capacity=rng.choice((1, 2)) if 2 * tokens <= MAX_TOKENS else 1,
                    plan=rng.randint(1, 1 << 20))


def _plan(case):
    """[layer][unit] plans of both kinds; the same for every seed, so that the work of a case is known."""
    shape, rng = MODELS[case["model"]].with_layers(case["layers"]), random.Random(case["plan"])
    bits, share = BIT_MIXES[case["bits"]]
    grids = []
    for n_units in (shape.n_heads, shape.n_ffn_slices):
        grid = []
        for layer in range(shape.n_layers):
            kept = set(rng.sample(range(n_units), max(1, round(case["keep"] * n_units))))
            grid.append([UnitPlan(i in kept, rng.choices(bits, share)[0], layer < case["resident"]) for i in range(n_units)])
        grids.append(grid)
    return shape, grids[0], grids[1]


def _lens(case):
    """Valid tokens of each sequence of a ragged batch: between a quarter and all of the padded length."""
    rng = random.Random(case["plan"] + 1)
    return [case["seq"]] + [rng.randint((case["seq"] + 3) // 4, case["seq"]) for _ in range(case["batch"] - 1)]


def _table(bits):
    """Means of the 2**bits equal-population slices of N(0, STD**2)."""
    normal, n = NormalDist(), 1 << bits
    density = [0.0] + [normal.pdf(normal.inv_cdf(c / n)) for c in range(1, n)] + [0.0]
    return np.array([(density[c] - density[c + 1]) * n * STD for c in range(n)], dtype=np.float32)


_TABLES = {bits: _table(bits) for bits in (2, 3, 4, 5, 6)}


def _blob(rng, bits, n):
    if bits == 32:
        weights = rng.standard_normal(n, dtype=np.float32) * np.float32(STD)
        return ShardBlob(32, weights.view(np.uint32), None, np.zeros(0, np.uint32), np.zeros(0, np.float32))
    words = np.frombuffer(rng.bytes(n * bits // 8), dtype=np.uint32)
    table = _TABLES[bits] * np.float32(rng.uniform(0.9, 1.1))
    off = np.unique(rng.integers(0, n, round(TAILS * n), dtype=np.uint32))
    return ShardBlob(bits, words, table, off, rng.standard_normal(off.size, dtype=np.float32) * np.float32(10 * STD))


def _dense(rng, shape):
    def n(*dims):
        return rng.standard_normal(dims, dtype=np.float32) * np.float32(STD)

    d, heads, slices = shape.hidden, shape.n_heads, shape.n_ffn_slices
    return {"bq": n(heads, shape.head_dim), "bk": n(heads, shape.head_dim), "bv": n(heads, shape.head_dim), "bo": n(d),
            "b1": n(slices, shape.slice_width), "b2": n(d), "ln1_g": 1 + n(d), "ln1_b": n(d), "ln2_g": 1 + n(d), "ln2_b": n(d)}


_streams = {}


def _stream():
    """The stream a program runs its model on: forwards follow one another, whichever plan they belong to."""
    device = torch.cuda.current_device()
    if device not in _streams:
        _streams[device] = torch.cuda.Stream()
    return _streams[device].cuda_stream


class _Forward:
    def __init__(self, case, seed):
        self.session = None
        shape, attn, ffn = _plan(case)
        rng = np.random.Generator(np.random.PCG64(seed))
        blobs = {(layer, kind, i): _blob(rng, u.bits, unit_weight_count(shape, kind))
                 for layer in range(shape.n_layers) for kind, grid in ((ATTN, attn), (FFN, ffn)) for i, u in enumerate(grid[layer]) if u.keep}
        work = SimpleNamespace(shape=shape, batch=case["batch"], seq=case["seq"], act_dtype=case["dtype"], ln_eps=1e-12,
                               ring_slots=case["slots"], attn_plan=attn, ffn_plan=ffn, blobs=blobs,
                               dense=[_dense(rng, shape) for _ in range(shape.n_layers)])
        self.case, self.batch, self.seq, host = case, case["batch"], case["seq"], case["entry"] == "host"
        gen = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.randn((self.batch, self.seq, shape.hidden), generator=gen, device="cuda")
        x = x.bfloat16() if case["dtype"] == "bf16" else x
        lens = torch.tensor(_lens(case), dtype=torch.int32) if case["ragged"] else None
        if host:
            self.x, self.y = x.cpu().pin_memory(), torch.zeros(x.shape, dtype=x.dtype).pin_memory()
            self.lens = lens.pin_memory() if case["ragged"] else None
        else:
            self.x, self.y, self.lens = x, torch.zeros_like(x), lens.cuda() if case["ragged"] else None
        self.lens_at = self.lens.data_ptr() if case["ragged"] else 0
        torch.cuda.synchronize()
        self.session = sti.Session(work, device=torch.cuda.current_device(), compute_stream=_stream(), max_batch=self.batch * case["capacity"])

    def __del__(self):
        if self.session is not None:
            self.session.close()

    def run(self):
        plan, x, y = self.session.plan, self.x.data_ptr(), self.y.data_ptr()
        if self.case["entry"] == "layer":
            sti.sti_layer_forward(plan, 0, x, y, self.batch, self.seq, self.lens_at)
        elif self.case["entry"] == "device":
            sti.sti_model_forward(plan, x, y, self.batch, self.seq, self.lens_at)
        else:        # the result is read on the host, so the program waits for it
            sti.sti_model_forward_host(plan, x, y, self.batch, self.seq, self.lens_at)
            sti.sti_sync(self.session.ctx)
        return self.y


class _Quantize:
    def __init__(self, case, seed):
        units, n, self.bits = case["units"], case["weights"], case["bits"]
        gen = torch.Generator(device="cuda").manual_seed(seed)
        self.w = torch.randn((units, n), generator=gen, device="cuda").mul_(STD)
        # heavier tails on a part of the weights, as in trained models
        self.w[torch.rand((units, n), generator=gen, device="cuda") < TAILS] *= 10
        self.units, self.n, self.max_out = units, n, n // 64
        self.codes = torch.zeros((units, n * self.bits // 32), dtype=torch.int32, device="cuda")
        self.centroids = torch.zeros((units, 1 << self.bits), device="cuda")
        self.off = torch.zeros((units, self.max_out), dtype=torch.int32, device="cuda")
        self.val = torch.zeros((units, self.max_out), device="cuda")
        self.count = torch.zeros(units, dtype=torch.int32, device="cuda")
        self.workspace = torch.empty(sti.sti_quantize_workspace_bytes(units, n), dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()

    def run(self):
        sti.sti_quantize_units(self.w.data_ptr(), self.units, self.n, self.bits, self.codes.data_ptr(), self.centroids.data_ptr(),
                               self.off.data_ptr(), self.val.data_ptr(), self.max_out, self.count.data_ptr(), self.workspace.data_ptr(),
                               self.workspace.numel(), device=torch.cuda.current_device(), stream=torch.cuda.current_stream().cuda_stream)
        return {"codes": self.codes, "centroids": self.centroids, "outlier_offsets": self.off, "outlier_values": self.val, "outliers": self.count}


def prepare(case, seed):
    return _Forward(case, seed) if case["kind"] == "forward" else _Quantize(case, seed)


def run(state):
    return state.run()


def work(case):
    if case["kind"] == "quantize":
        n, bits = case["units"] * case["weights"], case["bits"]
        # the weights in; the index stream, the tables and (0.2 % with the normal ones) the outlier pairs out.  The
        # arithmetic that any method needs: the fit's two sums, and finding each weight's cluster among 2**bits.
        return {"bytes": n * 4 + n * bits / 8 + case["units"] * ((1 << bits) * 4 + 4) + 0.002 * n * 8, "flops": n * (4.0 + bits)}
    shape, attn, ffn = _plan(case)
    tokens, d = case["batch"] * case["seq"], shape.hidden
    pairs = case["seq"] * (sum(_lens(case)) if case["ragged"] else tokens)        # (query, valid key) pairs of one head
    size, flops = 2 * tokens * d * (2 if case["dtype"] == "bf16" else 4), 0.0
    for layer in range(shape.n_layers):
        for kind, grid in ((ATTN, attn), (FFN, ffn)):
            n = unit_weight_count(shape, kind)
            for u in grid[layer]:
                if u.keep:
                    size += n * u.bits / 8 + (0 if u.bits == 32 else (4 << u.bits) + 8 * TAILS * n)
                    flops += 2.0 * tokens * n + (4.0 * pairs * shape.head_dim if kind == ATTN else 0.0)
        size += 4 * (3 * shape.n_heads * shape.head_dim + shape.ffn + 6 * d)
    return {"bytes": size, "flops": flops}


def tolerance(case):
    if case["kind"] == "quantize":
        return {"rel": 1e-6, "max": 1e-5, "differ": 0.0}        # streams, offsets and counts whole; centroids are rounded fp64 means
    return {"rel": 1e-2}        # bf16 operands, fp32 accumulation
