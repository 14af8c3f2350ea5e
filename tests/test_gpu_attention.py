"""Attention against the oracle layer in each shape of the mma.sync kernel (query tiles, key splits, key blocks) and where the
tensor-core kernel takes over, at
lengths around the block sizes, with and without padding masks."""
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


@pytest.mark.parametrize("batch,seq,masked", [
    (1, 1, False), (3, 17, True), (2, 32, True),             # up to 32 keys: one block of 32
    (2, 33, True), (1, 64, False),                           # up to 64: tiles of 64 queries
    (1, 65, False), (2, 97, True), (1, 128, True),           # few CTAs: 32 queries, keys split in two
    (1, 129, True), (2, 200, True), (1, 256, False),         # ... and in four
    (10, 150, True), (8, 300, True), (6, 256, True),         # 64 queries, keys split in two; what the O projection leaves
    (17, 150, True), (17, 190, True), (25, 100, True),       # 128 queries, blocks of 32 and of 64 keys
    (50, 70, True), (60, 64, False),                         # more tiles of 128 queries than SMs: 32- and 64-key blocks
    (50, 97, True), (50, 128, True), (17, 385, True),        # ... from 97 keys on the tensor-core kernel
])
def test_attention_shapes(batch, seq, masked):
    from gpu_util import run_layer, rel_err, REL_TOL
    shape = W.ModelShape(n_layers=1, hidden=256, n_heads=4, head_dim=64, ffn=1024, n_ffn_slices=4)
    attn = [[W.UnitPlan(i != 1, 4, True) for i in range(4)]]
    ffn = [[W.UnitPlan(True, 4, True) for _ in range(4)]]
    work = W.build_workload("attention", shape, batch, seq, "f32", attn, ffn, seed=batch * 1000 + seq)
    lens = np.random.default_rng(seq).integers(1, seq + 1, batch).tolist() if masked else None
    if masked:
        lens[0] = min(seq, 1 + 64 * (seq // 64))             # one key into the last block
    a, f = O.decode_layer(work, 0)
    ref = O.layer_forward(work.x, work.dense[0], a, f, eps=work.ln_eps, seq_lens=lens)
    with sti.Session(work) as s:
        y = run_layer(s, work, 0, lens=lens)
    assert np.isfinite(y).all()
    assert rel_err(y, ref) <= REL_TOL


@pytest.mark.parametrize("batch,seq", [(2, 40), (3, 128), (3, 441), (50, 97), (50, 130), (26, 256), (17, 385)])   # the last four: tensor cores
def test_sequences_without_a_valid_key(batch, seq):
    """Their attention contributes nothing, whatever the buffers held before; the others are not affected."""
    from gpu_util import run_layer, rel_err, REL_TOL
    shape = W.ModelShape(n_layers=1, hidden=256, n_heads=4, head_dim=64, ffn=1024, n_ffn_slices=4)
    attn = [[W.UnitPlan(i != 1, 4, True) for i in range(4)]]
    ffn = [[W.UnitPlan(True, 4, True) for _ in range(4)]]
    work = W.build_workload("empty", shape, batch, seq, "f32", attn, ffn, seed=batch + seq)
    lens = [0 if b % 2 else 1 + (7 * b) % seq for b in range(batch)]
    a, f = O.decode_layer(work, 0)
    with sti.Session(work) as s:
        poison = torch.full((batch, seq, shape.hidden), float("nan"), device="cuda")
        run_layer(s, work, 0, poison)                        # every row of the attention output holds NaN
        y = run_layer(s, work, 0, lens=lens)
    for b in range(batch):
        ref = O.layer_forward(work.x[b:b + 1], work.dense[0], a if lens[b] else {}, f, eps=work.ln_eps, seq_lens=lens[b:b + 1])
        assert rel_err(y[b], ref[0]) <= REL_TOL, (b, lens[b])


@pytest.mark.parametrize("batch,seq,act", [(2, 40, "f32"), (3, 130, "bf16"),                       # mma.sync
                                           (50, 97, "f32"), (50, 130, "bf16"), (26, 250, "f32"), (17, 441, "bf16")])   # tensor cores
def test_padding_does_not_reach_valid_rows(batch, seq, act):
    """Every padded row of the input is NaN, every third sequence has nothing else: the valid rows are those of an input without
    them.  Odd sequence lengths put the next sequence's rows into the last group of 16 keys."""
    from gpu_util import run_layer, to_device_act, rel_err, REL_TOL
    shape = W.ModelShape(n_layers=1, hidden=256, n_heads=4, head_dim=64, ffn=1024, n_ffn_slices=4)
    attn = [[W.UnitPlan(i != 1, 4, True) for i in range(4)]]
    ffn = [[W.UnitPlan(True, 4, True) for _ in range(4)]]
    work = W.build_workload("padding", shape, batch, seq, act, attn, ffn, seed=batch + seq)
    # full length, one key past a group of 16, one short of it, anything; empty
    lens = [0 if b % 3 == 1 else (seq, min(seq, 16 * (1 + b // 3) + 1), max(1, seq - seq % 16 - 1), 1 + 31 * b % seq)[b % 4] for b in range(batch)]
    x, clean = to_device_act(work), work.x.copy()
    for b, n in enumerate(lens):
        x[b, n:] = float("nan")
        clean[b, n:] = 0.0
    a, f = O.decode_layer(work, 0)
    with sti.Session(work) as s:
        y = run_layer(s, work, 0, x, lens=lens)
    for b, n in enumerate(lens):
        if n:
            ref = O.layer_forward(clean[b:b + 1], work.dense[0], a, f, eps=work.ln_eps, seq_lens=[n])
            assert np.isfinite(y[b, :n]).all(), (b, n)
            assert rel_err(y[b, :n], ref[0, :n]) <= REL_TOL, (b, n)
