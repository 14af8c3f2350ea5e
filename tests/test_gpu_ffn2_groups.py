"""How FFN2's K range is cut follows the call's token count, not what the context could take: a call gives the same bytes in a
context sized for it and in larger ones, and calls of different sizes through one plan match the oracle."""
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


def _work(batch, seq, kept):
    shape = W.ModelShape(n_layers=1, hidden=768, n_heads=4, head_dim=64, ffn=3072, n_ffn_slices=12)
    attn = [[W.UnitPlan(True, 3, True) for _ in range(4)]]
    ffn = [[W.UnitPlan(i < kept, 2 + i % 5, True) for i in range(12)]]
    return W.build_workload("ffn2_groups", shape, batch, seq, "f32", attn, ffn, seed=kept)


@pytest.mark.parametrize("batch,seq,kept", [(1, 128, 12), (1, 77, 9), (3, 100, 12), (8, 128, 9)])
def test_the_context_s_capacity_does_not_change_a_call(batch, seq, kept):
    from gpu_util import run_layer
    work, outs = _work(batch, seq, kept), []
    for max_batch in (batch, 8 * batch, 4200 // seq + 1):        # the largest takes FFN2 in one plane in its own largest calls
        with sti.Session(work, max_batch=max_batch) as s:
            outs.append(run_layer(s, work, 0))
    assert np.array_equal(outs[0], outs[1]) and np.array_equal(outs[0], outs[2])


def test_calls_of_all_sizes_through_one_plan():
    from gpu_util import from_device_act, rel_err, REL_TOL
    seq, most = 127, 20                                          # up to 2,540 tokens
    work = _work(most, seq, 12)
    a, f = O.decode_layer(work, 0)
    ref = O.layer_forward(work.x, work.dense[0], a, f, eps=work.ln_eps)
    x = torch.from_numpy(work.x_dev).cuda()
    with sti.Session(work) as s:
        for batch in (1, 20, 2, 8, 5, 9, 13):
            y = torch.full_like(x[:batch], float("nan"))
            torch.cuda.synchronize()
            sti.sti_layer_forward(s.plan, 0, x.data_ptr(), y.data_ptr(), batch, seq, 0)
            sti.sti_sync(s.ctx)
            assert rel_err(from_device_act(y), ref[:batch]) <= REL_TOL, batch
