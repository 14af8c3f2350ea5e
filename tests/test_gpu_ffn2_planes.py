"""FFN2 of calls of many tokens in one plane of fp32 sums and in several (K splits that the LayerNorm adds up), inside a whole layer:
against the oracle layer and against one another, on token counts that give whole and ragged pairs of token tiles and one or many tiles
per pair of CTAs."""
import os

import numpy as np
import pytest
import torch

import workloads as W
from oracle import sti_oracle as O

pytestmark = pytest.mark.gpu

sti = pytest.importorskip("paper_2207_05022_b200")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2207_05022_b200 import build
    build.build_library()
    sti.load_library()


def _work(batch, seq, act, seed, keep=lambda i: True):
    shape = W.ModelShape(n_layers=1, hidden=256, n_heads=4, head_dim=64, ffn=1536, n_ffn_slices=6)
    bits = [2, 3, 4, 5, 6, 32]
    attn = [[W.UnitPlan(True, bits[i % 5], True) for i in range(4)]]
    ffn = [[W.UnitPlan(keep(i), bits[(i + 1) % 6], True) for i in range(6)]]
    return W.build_workload("planes", shape, batch, seq, act, attn, ffn, seed=seed, outlier_stress=0.0015)


def _run(work, tune):
    from gpu_util import run_layer
    old = os.environ.get("STI_TUNE")
    os.environ["STI_TUNE"] = tune
    try:
        with sti.Session(work) as s:
            y = run_layer(s, work, 0)
            launches = sti.sti_ctx_launch_count(s.ctx)
        return y, launches
    finally:
        if old is None:
            os.environ.pop("STI_TUNE", None)
        else:
            os.environ["STI_TUNE"] = old


@pytest.mark.parametrize("batch,seq,act,budget,splits,keep", [
    (16, 128, "bf16", 148, 4, lambda i: True),     # 2,048 tokens: eight tile pairs, one tile or none per CTA pair
    (16, 128, "f32", 4, 2, lambda i: True),        # two CTA pairs: several tiles each
    (11, 100, "bf16", 4, 3, lambda i: i != 4),     # 1,100 tokens: nine tiles (odd), ragged rows, five slices
    (24, 128, "bf16", 8, 4, lambda i: i % 2 == 0),      # 3,072 tokens, three slices: splits of three chunks
    (16, 128, "bf16", 148, 4, lambda i: i == 3),        # one slice kept: a single chunk per split
    (16, 128, "f32", 4, 3, lambda i: i in (0, 5)),      # two slices: eight chunks in three splits
])
def test_layer_with_one_and_with_several_planes(batch, seq, act, budget, splits, keep):
    from gpu_util import rel_err, REL_TOL
    work = _work(batch, seq, act, seed=batch * 100 + seq, keep=keep)
    a, f = O.decode_layer(work, 0)
    ref = O.layer_forward(work.x, work.dense[0], a, f, eps=work.ln_eps)
    y_1, _ = _run(work, f"f2_one_plane_min_tokens=1024,cta_budget={budget}")
    y_n, _ = _run(work, f"f2_one_plane_min_tokens=0,wide_splits={splits},cta_budget={budget}")
    assert rel_err(y_1, ref) <= REL_TOL
    assert rel_err(y_n, ref) <= REL_TOL
    # same bf16 products, fp32 sums in a different order: the two agree far below the tolerance
    # (bf16 outputs may differ by one rounding step of 2^-8 relative)
    assert rel_err(y_1, y_n.astype(np.float64)) <= (1e-2 if act == "bf16" else 2e-3)
