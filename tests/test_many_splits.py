"""Merge of sequences with more than 32 KV splits: 33 (the fewest), whole and ragged batches of 16, more than the 256 of one trip, beside
sequences with few splits or one; 16-bit and fp32 partials, bf16 and fp32 results."""
import numpy as np
import pytest

from paper_2605_10380_b200 import workloads as W
from tests.plan_util import plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,hq,d,lengths,q,lean", [
    ("bf16", 4, 128, [33 * 64 - 1], 1, "1"), ("bf16", 4, 128, [48 * 64], 3, "1"), ("bf16", 8, 128, [7000], 2, "0"),
    ("bf16", 4, 128, [5000, 30, 700], 8, "0"), ("f32", 2, 64, [40 * 64], 2, "1"), ("f32", 2, 128, [18000, 100], 1, "1"),
])
def test_many_splits(dtype, hq, d, lengths, q, lean, monkeypatch):
    import oracle
    from tests.gpu_util import DeviceBatch, check_attention, oracle_pools_after_append
    monkeypatch.setenv("AGX_SMALL_MIN_SPLIT", "64")
    monkeypatch.setenv("AGX_MERGE_SMS", lean)
    w = W.make_attn_workload("many", sum(lengths), dtype, hq, 1, d, lengths, [q] * len(lengths), spare_pages=1)
    b = DeviceBatch(w)
    out, lse = b.attend_append()
    assert b.status() == 0
    again, _ = b.attend_append()
    assert (again == out).all()   # splits are added in order
    kp, vp = oracle_pools_after_append(w)
    ref, _ = oracle.attn_paged_batch(w.q_block, kp, vp, w.page_table, w.dtype, w.prefix_len, w.q_len, w.cu_q)
    check_attention(out, ref, "many")


@pytest.mark.parametrize("tokens,q,hq,hkv,kind,splits", [(9000, 1, 8, 2, "small1", 36), (9000, 8, 8, 2, "small2", 36), (12000, 1, 16, 2, "small1", 47), (12000, 8, 16, 2, "stream", 47),
                                                         (4058, 129, 8, 2, "tile", 33), (6200, 40, 8, 1, "tile", 49), (6200, 100, 6, 2, "tile", 50)])
def test_many_splits_of_each_kernel(tokens, q, hq, hkv, kind, splits, monkeypatch):
    """fp32 rows of the small-q kernels and the one-Q-tile schedule, fp16 rows in tiles of the 256-row schedule."""
    import oracle
    from tests.gpu_util import DeviceBatch, check_attention, oracle_pools_after_append
    if kind == "tile":
        monkeypatch.setenv("AGX_TILE_SPLIT_TOKENS", "128")
        monkeypatch.setenv("AGX_STREAM_MAX_ROWS", "32")
    ln, = plan([tokens], [q], hq, hkv).launches
    assert ln.kind == kind and ln.seqs[0].nsplit == splits
    w = W.make_attn_workload("many", tokens, "bf16", hq, hkv, 128, [tokens], [q], spare_pages=1)
    b = DeviceBatch(w)
    out, lse = b.attend_append()
    assert b.status() == 0
    again, _ = b.attend_append()
    assert (again == out).all()
    kp, vp = oracle_pools_after_append(w)
    ref, ref_lse = oracle.attn_paged_batch(w.q_block, kp, vp, w.page_table, w.dtype, w.prefix_len, w.q_len, w.cu_q)
    check_attention(out, ref, "many")
    assert np.abs(lse - ref_lse).max() <= 5e-6   # (as in test_few_splits.py)
