"""Host steps read their pinned inputs in the stream's order, whatever in front of them writes these."""
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
    """Two handles take turns on one stream, with 20 other streams used before."""
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


def on_device(pinned):
    """The same memory as a CUDA tensor: pinned memory is mapped into the device's address space."""
    import torch

    class View:
        __cuda_array_interface__ = {"shape": tuple(pinned.shape), "typestr": "<i2", "data": (pinned.data_ptr(), False), "version": 3}
    t = torch.as_tensor(View(), device="cuda").view(pinned.dtype)
    assert t.data_ptr() == pinned.data_ptr()
    return t


@pytest.mark.parametrize("front", ["host_step", "attention", "callers_kernel"])
@pytest.mark.parametrize("between", [0, 1, 3])
def test_queries_written_further_in_front(front, between):
    """A long call writes the pinned queries, short attention calls of the library with other outputs follow, then comes the host step."""
    import torch

    from tests.gpu_util import DeviceBatch
    q = 8
    make = lambda name, P: W.make_attn_workload(name, P, "bf16", 32, 8, 128, [P], [q], spare_pages=1)  # noqa: E731
    long, short, last = make("long", 30000), make("short", 40), make("last", 700)
    pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).view(torch.bfloat16).pin_memory()  # noqa: E731
    results = []
    for wait in (True, False):
        a, b, c = DeviceBatch(long), DeviceBatch(short), DeviceBatch(last)
        x, out = (torch.zeros(q, 32, 128, dtype=torch.bfloat16).pin_memory() for _ in range(2))
        inputs = [pin(v) for w in (long, last) for v in (w.q_block, w.k_new, w.v_new)]
        ws = [torch.empty(t.h.verify_step_host_workspace_bytes(t.w.prefix_len, t.w.q_len, "bf16", 0, 0), dtype=torch.uint8, device="cuda") for t in (a, c)]
        big = torch.randn(1 << 28, device="cuda")
        step = lambda t, q_in, k, v, o, space: t.h.verify_step_host(t.k_pool, t.v_pool, t.page_table, t.w.prefix_len, t.w.q_len, q_in, k, v,  # noqa: E731
                                                                    None, "bf16", 0, 0, None, o, None, None, None, space, enqueue_only=True)
        done = lambda: torch.cuda.synchronize() if wait else None  # noqa: E731
        torch.cuda.synchronize()
        if front == "host_step":
            step(a, *inputs[:3], x, ws[0])
        elif front == "attention":
            a.h.attn_prefixed(a.q_block, a.k_pool, a.v_pool, a.page_table, long.prefix_len, long.q_len, on_device(x), None, a.ws)
        else:
            big.mul_(0.5)
            torch.mul(a.q_block, 2, out=on_device(x))
        done()
        for _ in range(between):
            b.h.attn_prefixed(b.q_block, b.k_pool, b.v_pool, b.page_table, short.prefix_len, short.q_len, b.out, None, b.ws)
        done()
        step(c, x, inputs[4], inputs[5], out, ws[1])
        torch.cuda.synchronize()
        assert a.status() == 0 and b.status() == 0 and c.status() == 0
        results.append((x.clone(), out.clone()))
    for i in (0, 1):
        assert torch.equal(results[0][i].view(torch.int16), results[1][i].view(torch.int16))
    assert bool(results[0][0].any())
