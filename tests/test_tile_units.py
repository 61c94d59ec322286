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
