"""Tensor-core schedules over few KV tiles: units of work (KV tile x Q tile) at the start and the end of the pipeline, a second Q
tile that is all padding, last tiles of every page count."""
import pytest

from paper_2605_10380_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split_tokens", ["0", "128", "384"])
@pytest.mark.parametrize("q,hq,hkv", [(97, 32, 8), (129, 8, 8), (200, 24, 8), (8, 32, 8)], ids=["short_last_chunk", "one_row_in_b", "two_chunks", "stream"])
def test_few_kv_tiles(q, hq, hkv, split_tokens, monkeypatch):
    from tests.gpu_util import DeviceBatch, check_attention, oracle_pools_after_append
    import oracle
    monkeypatch.setenv("AGX_TILE_SPLIT_TOKENS", split_tokens)
    monkeypatch.setenv("AGX_STREAM_MIN_TOKENS", "0")
    monkeypatch.setenv("AGX_STREAM_MAX_ROWS", "32")
    P = [0, 1, 31, 120, 128, 250, 384, 500, 767]
    w = W.make_attn_workload("units", 3 * q + hq, "bf16", hq, hkv, 128, P, [q] * len(P), spare_pages=2)
    b = DeviceBatch(w)
    out, _ = b.attend_append()
    assert b.status() == 0
    kp, vp = oracle_pools_after_append(w)
    ref, _ = oracle.attn_paged_batch(w.q_block, kp, vp, w.page_table, w.dtype, w.prefix_len, w.q_len, w.cu_q)
    check_attention(out, ref, "units")


SCHEDULES = [("stream", 8, "0"), ("tile", 130, "0"), ("tile_split", 130, "128")]


def _batch(q, split_tokens, P, monkeypatch):
    from tests.gpu_util import DeviceBatch
    monkeypatch.setenv("AGX_TILE_SPLIT_TOKENS", split_tokens)
    monkeypatch.setenv("AGX_STREAM_MIN_TOKENS", "0")
    return DeviceBatch(W.make_attn_workload("columns", P + q, "bf16", 32, 8, 128, [P], [q], spare_pages=1))


@pytest.mark.parametrize("column", [0, 1, 2, 15, 16, 17, 127])
@pytest.mark.parametrize("name,q,split_tokens", SCHEDULES, ids=[s[0] for s in SCHEDULES])
def test_a_nan_in_one_key_reaches_every_row_whatever_its_column(name, q, split_tokens, column, monkeypatch):
    """(the columns of a KV tile take their exponentials from two different units)"""
    import torch
    b = _batch(q, split_tokens, 500, monkeypatch)
    tok, g = 128 + column, 3
    b.k_pool[int(b.w.page_table[0, tok // 16]), g, tok % 16, 77] = float("nan")
    b.attend_append()
    nan = torch.isnan(b.out).all(dim=-1)
    assert bool(nan[:, 4 * g:4 * g + 4].all()) and not bool(nan[:, :4 * g].any()) and not bool(nan[:, 4 * g + 4:].any())


@pytest.mark.parametrize("column", [0, 1, 2, 15, 16, 17, 127])
@pytest.mark.parametrize("name,q,split_tokens", SCHEDULES, ids=[s[0] for s in SCHEDULES])
def test_a_hidden_token_weighs_nothing_whatever_its_column(name, q, split_tokens, column, monkeypatch):
    """The last token of the block, at each column, is hidden from all rows but the last: how large its V is changes no bit of them."""
    import torch
    P = 512 + column + 1 - q
    outs = []
    for value in (1.0, 3e38):
        b = _batch(q, split_tokens, P, monkeypatch)
        b.v_new[q - 1] = value
        b.attend_append()
        outs.append((b.out, b.lse))
    assert torch.equal(outs[0][0][:q - 1], outs[1][0][:q - 1]) and torch.equal(outs[0][1][:q - 1], outs[1][1][:q - 1])
    assert not torch.equal(outs[0][0][q - 1], outs[1][0][q - 1])
