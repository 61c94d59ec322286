"""Host steps read their pinned inputs ahead of the stream's order, except what the handle's call in front writes."""
import numpy as np
import pytest

from paper_2605_10380_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,q", [(40, 1), (1000, 8), (3000, 8), (700, 40)], ids=["no_split", "splits", "many_splits", "stream"])
def test_results_of_one_step_are_the_queries_of_the_next(P, q):
    import torch

    from tests.gpu_util import DeviceBatch
    w = W.make_attn_workload("chain", P + q, "bf16", 32, 8, 128, [P], [q], spare_pages=1)
    pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).view(torch.bfloat16).pin_memory()  # noqa: E731
    steps = 12
    results = []
    for wait in (True, False):   # each step waited for, and all of them at once
        b = DeviceBatch(w)
        k, v = pin(w.k_new), pin(w.v_new)
        bufs = [pin(w.q_block)] + [torch.zeros(w.total_q, 32, 128, dtype=torch.bfloat16).pin_memory() for _ in range(steps)]
        ws = torch.empty(b.h.verify_step_host_workspace_bytes(w.prefix_len, w.q_len, "bf16", 0, 0), dtype=torch.uint8, device="cuda")
        for i in range(steps):
            b.h.verify_step_host(b.k_pool, b.v_pool, b.page_table, w.prefix_len, w.q_len, bufs[i], k, v, None, "bf16", 0, 0, None, bufs[i + 1],
                                 None, None, None, ws, enqueue_only=not wait)
        torch.cuda.synchronize()
        assert b.status() == 0
        results.append(torch.stack(bufs).clone())
    assert torch.equal(results[0].view(torch.int16), results[1].view(torch.int16))


@pytest.mark.parametrize("P,q", [(40, 1), (1000, 8), (700, 40)], ids=["no_split", "splits", "stream"])
def test_results_of_one_handle_are_the_queries_of_another(P, q):
    """Two handles take turns on one stream, with 20 other streams used before (more than are remembered)."""
    import torch

    from tests.gpu_util import DeviceBatch
    w = W.make_attn_workload("turns", P + q, "bf16", 32, 8, 128, [P], [q], spare_pages=1)
    pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).view(torch.bfloat16).pin_memory()  # noqa: E731
    steps = 12
    results = []
    for wait in (True, False):
        two = [DeviceBatch(w), DeviceBatch(w)]
        for _ in range(0 if wait else 20):
            with torch.cuda.stream(torch.cuda.Stream()):
                two[0].attend()
        torch.cuda.synchronize()
        k, v = pin(w.k_new), pin(w.v_new)
        bufs = [pin(w.q_block)] + [torch.zeros(w.total_q, 32, 128, dtype=torch.bfloat16).pin_memory() for _ in range(steps)]
        ws = [torch.empty(b.h.verify_step_host_workspace_bytes(w.prefix_len, w.q_len, "bf16", 0, 0), dtype=torch.uint8, device="cuda") for b in two]
        for i in range(steps):
            b = two[i % 2]
            b.h.verify_step_host(b.k_pool, b.v_pool, b.page_table, w.prefix_len, w.q_len, bufs[i], k, v, None, "bf16", 0, 0, None, bufs[i + 1],
                                 None, None, None, ws[i % 2], enqueue_only=not wait)
        torch.cuda.synchronize()
        assert two[0].status() == 0 and two[1].status() == 0
        results.append(torch.stack(bufs).clone())
    assert torch.equal(results[0].view(torch.int16), results[1].view(torch.int16))
