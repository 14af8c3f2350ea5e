"""The LayerNorm kernels against the oracle layer at row counts around the lines between them (2048, sixteen rows per SM,
4096), with ragged row counts that leave a last CTA partly empty."""
import pytest

import workloads as W
from oracle import sti_oracle as O

pytestmark = pytest.mark.gpu

sti = pytest.importorskip("paper_2207_05022_b200")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2207_05022_b200 import build
    build.build_library()
    sti.load_library()


@pytest.mark.parametrize("batch,seq,act", [
    (23, 89, "bf16"), (16, 128, "f32"), (19, 109, "bf16"),        # 2047, 2048, 2071 rows
    (37, 64, "bf16"), (103, 23, "f32"),                           # 2368, 2369
    (63, 65, "bf16"), (64, 64, "f32"), (57, 73, "bf16"),          # 4095, 4096, 4161
])
def test_layernorm_rows(batch, seq, act):
    from gpu_util import run_layer, rel_err, REL_TOL
    shape = W.ModelShape(n_layers=1, hidden=256, n_heads=4, head_dim=64, ffn=1024, n_ffn_slices=4)
    attn = [[W.UnitPlan(True, 4, True) for _ in range(4)]]
    ffn = [[W.UnitPlan(True, 4, True) for _ in range(4)]]
    work = W.build_workload("layernorm", shape, batch, seq, act, attn, ffn, seed=batch * 1000 + seq)
    a, f = O.decode_layer(work, 0)
    ref = O.layer_forward(work.x, work.dense[0], a, f, eps=work.ln_eps)
    with sti.Session(work) as s:
        y = run_layer(s, work, 0)
    assert rel_err(y, ref) <= REL_TOL


@pytest.mark.parametrize("kept", [4, 5, 8, 9, 12])
def test_layernorm_planes(kept, monkeypatch):
    # one partial-sum plane per kept FFN slice: four, up to eight in one go, more in further steps
    from gpu_util import run_layer, rel_err, REL_TOL
    monkeypatch.setenv("STI_TUNE", "f2_group=1")
    shape = W.ModelShape(n_layers=1, hidden=256, n_heads=4, head_dim=64, ffn=3072, n_ffn_slices=12)
    attn = [[W.UnitPlan(True, 4, True) for _ in range(4)]]
    ffn = [[W.UnitPlan(i < kept, 4, True) for i in range(12)]]
    work = W.build_workload("planes", shape, 3, 37, "f32", attn, ffn, seed=kept)
    a, f = O.decode_layer(work, 0)
    ref = O.layer_forward(work.x, work.dense[0], a, f, eps=work.ln_eps)
    with sti.Session(work) as s:
        y = run_layer(s, work, 0)
    assert rel_err(y, ref) <= REL_TOL
