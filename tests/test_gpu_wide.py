"""GEMMs over the working buffer (calls of many tokens): each of a layer's four against an fp64 product of the decoded weights at
the edges of its tiles, and whole forwards, in which a layer is decoded beside the one before it, against the same layers
called one by one, where every layer is decoded by itself first: the same bytes."""
import os

import numpy as np
import pytest
import torch

import workloads as W
from oracle import sti_oracle as O
from workloads.shards import ATTN, FFN

pytestmark = pytest.mark.gpu

sti = pytest.importorskip("paper_2207_05022_b200")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2207_05022_b200 import build
    build.build_library()
    sti.load_library()


BITS6 = [2, 3, 4, 5, 6, 32]


def _decoded(sess, shape, kind, index, matrix):
    rows, cols = ((64, shape.hidden) if matrix < 3 else (shape.hidden, 64)) if kind == ATTN else \
        ((shape.slice_width, shape.hidden) if matrix == 0 else (shape.hidden, shape.slice_width))
    w = torch.zeros(rows, cols, dtype=torch.bfloat16, device="cuda")
    sti.sti_shard_decode(sess.plan, 0, kind, index, matrix, 0, 0, w.data_ptr())
    sti.sti_sync(sess.ctx)
    return w.double()


@pytest.mark.parametrize("nt,splits", [(256, 1), (128, 1), (256, 4), (128, 3)])
@pytest.mark.parametrize("tokens,heads,slices,hidden", [
    (1, 1, 1, 256),          # one token, one 64-column chunk of K in the O projection, 192 features in a 256-wide tile
    (33, 2, 3, 128),         # fewer rows than a store box, hidden narrower than a tile
    (129, 5, 2, 384),        # the pair's second CTA has one row
    (300, 3, 5, 256),        # two token pairs, the second one ragged
    (1000, 4, 4, 640),       # more tiles than one: accumulators alternate
])
def test_products_at_tile_edges(tokens, heads, slices, hidden, nt, splits, monkeypatch):
    monkeypatch.setenv("STI_TUNE", f"wide_nt={nt},wide_splits={splits},cta_budget=16")     # eight pairs: several tiles each
    shape = W.ModelShape(n_layers=1, hidden=hidden, n_heads=heads, head_dim=64, ffn=128 * slices, n_ffn_slices=slices)
    attn = [[W.UnitPlan(True, BITS6[i % 6], True) for i in range(heads)]]
    ffn = [[W.UnitPlan(True, BITS6[(i + 3) % 6], True) for i in range(slices)]]
    work = W.build_workload("wide", shape, 1, 8, "bf16", attn, ffn, seed=tokens)
    gen = torch.Generator(device="cuda").manual_seed(tokens)
    with sti.Session(work) as s:
        for gemm in range(4):
            if gemm == 0:
                w = torch.cat([_decoded(s, shape, ATTN, h, m) for h in range(heads) for m in range(3)])
            elif gemm == 1:
                w = torch.cat([_decoded(s, shape, ATTN, h, 3) for h in range(heads)], dim=1)
            else:
                w = torch.cat([_decoded(s, shape, FFN, j, gemm - 2) for j in range(slices)], dim=gemm - 2)
            n, k = w.shape
            x = torch.randn(tokens, k, generator=gen, device="cuda").bfloat16()
            sums = gemm in (1, 3)
            guard = 64                                     # elements behind the output that must stay as they are
            out = torch.full((8 * tokens * n + guard,), float("nan"), dtype=torch.float32 if sums else torch.bfloat16, device="cuda")
            torch.cuda.synchronize()
            parts = sti.sti_gemm_probe(s.plan, 0, gemm, x.data_ptr(), tokens, out.data_ptr(), (out.numel() - guard) * out.element_size(), 2)
            sti.sti_sync(s.ctx)
            assert torch.isnan(out[parts * tokens * n:]).all()
            got = out[:parts * tokens * n].double()
            if gemm == 0:
                got = got.view(3 * heads, tokens, 64).permute(1, 0, 2).reshape(tokens, n)
            else:
                got = got.view(parts, tokens, n).sum(0)
            want, scale = x.double() @ w.T, x.double().abs() @ w.abs().T
            # fp32 accumulation of k exact products: k roundings of 2^-24 of the sum of magnitudes; a bf16 result adds 2^-9 of itself, at most 2^-8 of the exact one
            bound = scale * k * 2.0 ** -24 + (0 if sums else want.abs() * 2.0 ** -8) + 1e-30
            assert ((got - want).abs() <= bound).all(), (gemm, parts)


def _layers(n, act, streamed_from):
    """A model with a layer that keeps no head, one that keeps no slice, and uncompressed units."""
    shape = W.ModelShape(n_layers=n, hidden=256, n_heads=4, head_dim=64, ffn=1024, n_ffn_slices=4)
    attn = [[W.UnitPlan(l != 2 and (l + i) % 4 != 1, BITS6[(l + i) % 6], l < streamed_from) for i in range(4)] for l in range(n)]
    ffn = [[W.UnitPlan(l != 4 and (l + i) % 3 != 1, BITS6[(2 * l + i) % 6], l < streamed_from) for i in range(4)] for l in range(n)]
    return W.build_workload("layers", shape, 5, 127, act, attn, ffn, seed=n, ring_slots=2)


@pytest.mark.parametrize("act,streamed_from", [("bf16", 99), ("f32", 99), ("bf16", 3), ("bf16", 0)])
def test_decoding_ahead_gives_the_same_bytes(act, streamed_from, monkeypatch):
    from gpu_util import from_device_act, rel_err, to_device_act, REL_TOL
    monkeypatch.setenv("STI_TUNE", "wide_min_tokens=1")
    work = _layers(7, act, streamed_from)
    x = to_device_act(work)
    with sti.Session(work) as s:
        cur = x.clone()
        for layer in range(7):
            y = torch.zeros_like(cur)
            torch.cuda.synchronize()
            sti.sti_layer_forward(s.plan, layer, cur.data_ptr(), y.data_ptr(), work.batch, work.seq, 0)
            sti.sti_sync(s.ctx)
            cur = y
        outs = [torch.full_like(x, float("nan")) for _ in range(4)]
        torch.cuda.synchronize()
        for o in outs:                                     # one after the other, not waited for in between
            sti.sti_model_forward(s.plan, x.data_ptr(), o.data_ptr(), work.batch, work.seq, 0)
        sti.sti_sync(s.ctx)
    for o in outs:
        assert torch.equal(o.view(torch.uint8), cur.view(torch.uint8))
    assert rel_err(from_device_act(cur), O.run_workload(work)) <= REL_TOL


@pytest.mark.parametrize("heads,slices", [
    ((2, 16, 16, 2, 2, 16), (2, 16, 16, 2, 2, 16)),        # two layers after a narrow one comes one that keeps all
    ((16, 16, 16, 1, 16, 16), (0, 16, 16, 0, 3, 16)),      # ... after one without a slice, whose O projection is its last product
    ((0, 16, 16, 0, 4, 16), (16, 16, 16, 2, 16, 16)),      # ... without a head
])
def test_layers_of_different_widths_give_the_same_bytes(heads, slices):
    """Layers decoded ahead while layers of other widths are still multiplied with, above the rule's threshold."""
    from gpu_util import from_device_act, rel_err, to_device_act, REL_TOL
    n = len(heads)
    shape = W.BERT_LARGE.with_layers(n)
    attn = [[W.UnitPlan(i < heads[l], BITS6[(l + i) % 5], True) for i in range(16)] for l in range(n)]
    ffn = [[W.UnitPlan(i < slices[l], BITS6[(2 * l + i) % 5], True) for i in range(16)] for l in range(n)]
    work = W.build_workload("widths", shape, 5, 128, "bf16", attn, ffn, seed=n, workers=4)
    x = to_device_act(work)
    with sti.Session(work) as s:
        cur = x.clone()
        for layer in range(n):
            y = torch.zeros_like(cur)
            torch.cuda.synchronize()
            sti.sti_layer_forward(s.plan, layer, cur.data_ptr(), y.data_ptr(), work.batch, work.seq, 0)
            sti.sti_sync(s.ctx)
            cur = y
        outs = [torch.full_like(x, float("nan")) for _ in range(20)]
        torch.cuda.synchronize()
        for o in outs:
            sti.sti_model_forward(s.plan, x.data_ptr(), o.data_ptr(), work.batch, work.seq, 0)
        sti.sti_sync(s.ctx)
    for o in outs:
        assert torch.equal(o.view(torch.uint8), cur.view(torch.uint8))
    assert rel_err(from_device_act(cur), O.run_workload(work)) <= REL_TOL


def test_forwards_behind_a_product_by_itself(monkeypatch):
    """Launched kernel by kernel: a forward decodes layer 1 ahead into the buffer in which a product queued just before it
    reads layer 3."""
    from gpu_util import to_device_act
    monkeypatch.setenv("STI_NO_GRAPH", "1")
    work = _layers(5, "bf16", 99)
    shape, T = work.shape, work.batch * work.seq
    x = to_device_act(work)
    planes = 3 * len(work.kept(3, ATTN))
    with sti.Session(work) as s:
        alone = torch.empty_like(x)
        sti.sti_model_forward(s.plan, x.data_ptr(), alone.data_ptr(), work.batch, work.seq, 0)
        rows = 16 * T                                      # a product that takes longer than the forward's first kernels
        act = torch.randn(rows, shape.hidden, device="cuda").bfloat16()
        want = torch.zeros(planes, rows, 64, dtype=torch.bfloat16, device="cuda")
        got = torch.zeros_like(want)
        torch.cuda.synchronize()
        sti.sti_gemm_probe(s.plan, 3, 0, act.data_ptr(), rows, want.data_ptr(), want.numel() * 2, 2)
        sti.sti_sync(s.ctx)
        for _ in range(10):
            y = torch.full_like(x, float("nan"))
            torch.cuda.synchronize()
            sti.sti_gemm_probe(s.plan, 3, 0, act.data_ptr(), rows, got.data_ptr(), got.numel() * 2, 2)
            sti.sti_model_forward(s.plan, x.data_ptr(), y.data_ptr(), work.batch, work.seq, 0)
            sti.sti_sync(s.ctx)
            assert torch.equal(got, want) and torch.equal(y, alone)


def test_the_rule_s_threshold_is_a_matter_of_the_call(monkeypatch):
    """Calls below and above the token count where the working buffer takes over, through one plan and interleaved."""
    from gpu_util import from_device_act, rel_err, to_device_act, REL_TOL
    work = _layers(7, "bf16", 99)
    ref = O.run_workload(work)
    x = to_device_act(work)
    with sti.Session(work) as s:
        for batch in (5, 1, 4, 3, 5, 2):
            y = torch.full_like(x[:batch], float("nan"))
            torch.cuda.synchronize()
            sti.sti_model_forward(s.plan, x.data_ptr(), y.data_ptr(), batch, work.seq, 0)
            sti.sti_sync(s.ctx)
            assert rel_err(from_device_act(y), ref[:batch]) <= REL_TOL, batch


@pytest.mark.parametrize("model,kept,context,calls", [
    ("large", 12, (1, 512), [(1, 400), (1, 488), (1, 385), (1, 512)]),
    ("large", 14, (8, 512), [(11, 134), (1, 512)]),
    ("base", 12, (8, 256), [(7, 251), (8, 256)]),
])
def test_calls_a_few_tokens_smaller_than_their_context(model, kept, context, calls):
    """Fewer tokens can take more planes of partial sums than the context's capacity does; fp32 activations, so that the residual
    that stands behind the planes is an fp32 copy."""
    from gpu_util import from_device_act, rel_err, REL_TOL
    shape = (W.BERT_BASE if model == "base" else W.BERT_LARGE).with_layers(1)
    attn = [[W.UnitPlan(i < kept, BITS6[i % 5], True) for i in range(shape.n_heads)]]
    ffn = [[W.UnitPlan(i < kept, BITS6[(i + 2) % 5], True) for i in range(shape.n_ffn_slices)]]
    work = W.build_workload("smaller", shape, 1, 8, "f32", attn, ffn, seed=kept)
    a, f = O.decode_layer(work, 0)
    with sti.Session(work, max_batch=context[0], max_seq=context[1]) as s:
        for batch, seq in calls:
            x = np.random.default_rng(seq).standard_normal((batch, seq, shape.hidden), dtype=np.float32)
            ref = O.layer_forward(x, work.dense[0], a, f, eps=work.ln_eps)
            x = torch.from_numpy(x).cuda()
            y = torch.full_like(x, float("nan"))
            torch.cuda.synchronize()
            sti.sti_layer_forward(s.plan, 0, x.data_ptr(), y.data_ptr(), batch, seq, 0)
            sti.sti_sync(s.ctx)
            assert rel_err(from_device_act(y), ref) <= REL_TOL, (batch, seq)


@pytest.mark.parametrize("layers,streamed,buffers", [(1, False, 1), (2, True, 1), (2, False, 2)])
def test_working_buffers_take_what_the_header_says(layers, streamed, buffers, monkeypatch):
    shape = W.BERT_LARGE.with_layers(layers)
    units = [[W.UnitPlan(True, 2, not streamed or l < 1) for _ in range(16)] for l in range(layers)]
    work = W.build_workload("memory", shape, 1, 512, "bf16", units, units, seed=layers, workers=layers)

    def taken(tune):
        monkeypatch.setenv("STI_TUNE", tune)
        with sti.Session(work, finalize=False) as s:
            before = torch.cuda.mem_get_info()[0]
            sti.sti_plan_finalize(s.plan)
            return before - torch.cuda.mem_get_info()[0]

    one = 2 * 16 * (unit_weights(shape, ATTN) + unit_weights(shape, FFN))
    extra = taken("wide_min_tokens=-1") - taken("wide_min_tokens=0")
    assert abs(extra - buffers * one) < 8 << 20            # planes of partial sums differ by up to 4 MB, allocations come in 2 MB


def unit_weights(shape, kind):
    return 4 * 64 * shape.hidden if kind == ATTN else 2 * shape.slice_width * shape.hidden
