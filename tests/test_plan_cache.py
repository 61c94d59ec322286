"""The handle keeps the launch plans of its last batches."""
import numpy as np
import pytest

from paper_2605_10380_b200 import workloads as W

pytestmark = pytest.mark.gpu


def test_the_layers_of_a_pipelined_host_step_plan_each_chunk_once(capfd, monkeypatch):
    import torch

    from tests.gpu_util import DeviceBatch
    monkeypatch.setenv("AGX_DEBUG_PLAN", "1")   # (a line for every plan that is made)
    w = W.make_attn_workload("layers", 17, "bf16", 32, 8, 128, [300], [900], spare_pages=1)
    b = DeviceBatch(w)
    pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).view(torch.bfloat16).pin_memory()  # noqa: E731
    q, k, v = pin(w.q_block), pin(w.k_new), pin(w.v_new)
    ws = torch.empty(b.h.verify_step_host_workspace_bytes(w.prefix_len, w.q_len, "bf16", 0, 0), dtype=torch.uint8, device="cuda")
    outs = [torch.zeros_like(q).pin_memory() for _ in range(3)]
    for out in outs:
        b.h.verify_step_host(b.k_pool, b.v_pool, b.page_table, w.prefix_len, w.q_len, q, k, v, None, "bf16", 0, 0, None, out, None, None, None, ws,
                             enqueue_only=True)
    torch.cuda.synchronize()
    assert b.status() == 0 and torch.equal(outs[0], outs[2])
    assert capfd.readouterr().err.count("agx plan: tile kernel") == 1 + 3   # the whole block (its workspace was asked for), 384 + 384 + 132 rows


def test_plans_of_other_batches_do_not_come_back_wrong():
    """More batches in turn than plans are kept, some of them equal but for one length."""
    import torch

    from tests.gpu_util import DeviceBatch
    w = W.make_attn_workload("turns", 18, "bf16", 32, 8, 128, [900, 40], [4, 2], spare_pages=1)
    one = DeviceBatch(w)
    one.append()
    lengths = [([900 - 16 * i, 40], [4, 2]) for i in range(20)] + [([900, 40], [3, 3]), ([900], [4])]
    ws = torch.empty(max(one.h.attn_workspace_bytes(*l) for l in lengths) + 256, dtype=torch.uint8, device="cuda")
    for P, Q in lengths * 2:
        fresh = DeviceBatch(w).h
        outs = [torch.zeros_like(one.q_block) for _ in range(2)]
        for h, out in zip((one.h, fresh), outs):
            h.attn_prefixed(one.q_block, one.k_pool, one.v_pool, one.page_table, P, Q, out, None, ws)
        assert torch.equal(*outs), (P, Q)
