"""The compiled argument marshalling: every form an argument may take gives the call the same arguments."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["list", "int64", "strided", "torch_cpu"])
@pytest.mark.parametrize("stream", ["none", "int", "object"])
def test_lengths_and_streams_in_every_form(form, stream):
    import torch

    from paper_2605_10380_b200 import workloads as W
    from tests.gpu_util import DeviceBatch
    w = W.make_attn_workload("binding", 31, "bf16", 32, 8, 128, [500, 33, 1200], [4, 1, 40], spare_pages=2)
    b = DeviceBatch(w)
    b.append()
    ref, _ = b.attend()
    lengths = []
    for a in (w.prefix_len, w.q_len):
        lengths.append({"list": a.tolist(), "int64": a.astype(np.int64), "strided": np.repeat(a, 2)[::2], "torch_cpu": torch.from_numpy(a)}[form])
    side = torch.cuda.Stream()
    out = torch.zeros_like(b.q_block)
    ws = torch.empty(max(256, b.h.attn_workspace_bytes(*lengths)), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    b.h.attn_prefixed(b.q_block, b.k_pool, b.v_pool, b.page_table, *lengths, out, None, ws,
                      stream={"none": None, "int": side.cuda_stream, "object": side}[stream])
    torch.cuda.synchronize()
    assert np.array_equal(out.double().cpu().numpy(), ref)


def test_arguments_that_are_none_or_of_the_wrong_type():
    import torch

    from paper_2605_10380_b200 import agx
    h = agx.Handle(32, 8, 128, "bf16")
    pool = torch.zeros(4, 8, 16, 128, dtype=torch.bfloat16, device="cuda")
    q = torch.zeros(1, 32, 128, dtype=torch.bfloat16, device="cuda")
    kv = torch.zeros(1, 8, 128, dtype=torch.bfloat16, device="cuda")
    table = torch.zeros(1, 4, dtype=torch.int32, device="cuda")
    with pytest.raises(agx.AgxError):
        h.attn_prefixed_append(q, None, kv, pool, pool, table, [5], [1], q)
    with pytest.raises(agx.AgxError):
        h.attn_prefixed(None, pool, pool, table, [5], [1], q)
    with pytest.raises(TypeError):
        h.attn_prefixed(q, np.zeros(4), pool, table, [5], [1], q)
    h.close()
    with pytest.raises(agx.AgxError):
        h.attn_prefixed(q, pool, pool, table, [5], [1], q)


@pytest.mark.parametrize("length", [32769, 32770, 32771, 16387, 2, 3])
def test_ngram_build_on_both_sides_of_the_one_launch_limit(length):
    """32768 windows is the largest stream built by one cluster; the table must not depend on which form built it."""
    import torch

    from oracle.toy_lm import build_ngram_table, ngram_drafts
    from paper_2605_10380_b200 import agx
    h = agx.Handle(32, 8, 128, "bf16")
    rng = np.random.default_rng(length)
    stream = rng.integers(0, 40, size=length).astype(np.int32)
    st = torch.from_numpy(stream).cuda()
    lut = torch.empty(agx.ngram_lut_bytes(length), dtype=torch.uint8, device="cuda")
    ws = torch.empty(agx.ngram_workspace_bytes(length), dtype=torch.uint8, device="cuda")
    h.ngram_build(st, 3, lut, ws)
    assert h.last_launch_count() == (1 if length - 2 <= 32768 else 3)
    table = build_ngram_table(stream.tolist(), 3)
    keys = list(table)[:500] + [(39, 41)]
    ctx = torch.tensor(keys, dtype=torch.int32, device="cuda")
    drafts = torch.zeros(len(keys), 4, dtype=torch.int32, device="cuda")
    has = torch.zeros(len(keys), dtype=torch.int32, device="cuda")
    h.ngram_draft(lut, ctx, torch.zeros_like(drafts), 4, drafts, has)
    torch.cuda.synchronize()
    for i, key in enumerate(keys):
        ref = ngram_drafts(table, list(key), 4, 3, fill=[0] * 4) if key in table else None
        assert has[i].item() == (ref is not None) and (ref is None or drafts[i].tolist() == ref)
