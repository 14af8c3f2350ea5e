"""Single layers called one right after the other (launched kernel by kernel beside the call before) give the same bytes as
with a wait after each call (one graph each): a chain in which every call reads what the one before wrote."""
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

sti = pytest.importorskip("paper_2207_05022_b200")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2207_05022_b200 import build
    build.build_library()
    sti.load_library()


@pytest.mark.parametrize("batch,seq,act", [(1, 1, "bf16"), (1, 128, "f32"), (4, 128, "bf16"), (27, 19, "bf16")])
def test_layer_chain(batch, seq, act):
    from gpu_util import to_device_act
    shape = W.ModelShape(n_layers=3, hidden=256, n_heads=4, head_dim=64, ffn=1024, n_ffn_slices=4)
    attn = [[W.UnitPlan(True, 2 + li + i % 2, True) for i in range(4)] for li in range(3)]
    ffn = [[W.UnitPlan(True, 6 - li, True) for _ in range(4)] for li in range(3)]
    work = W.build_workload("chain", shape, batch, seq, act, attn, ffn, seed=seq)
    with sti.Session(work) as s:
        def chain(wait):
            bufs = [to_device_act(work) for _ in range(13)]
            torch.cuda.synchronize()
            for i in range(12):
                sti.sti_layer_forward(s.plan, i % 3, bufs[i].data_ptr(), bufs[i + 1].data_ptr(), batch, seq, 0)
                if wait:
                    sti.sti_sync(s.ctx)
            sti.sti_sync(s.ctx)
            return bufs
        want = chain(True)
        for _ in range(4):
            got = chain(False)
            assert all(torch.equal(a.view(torch.uint8), b.view(torch.uint8)) for a, b in zip(want, got))
