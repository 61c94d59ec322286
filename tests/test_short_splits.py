"""Kernel for short KV splits with swapped MMA operands: 4, 8, 16 and 32 columns of query rows, one to three tiles of 128 tokens (the last
one short), splits merged through memory, in a cluster or not at all, blocks of one and of several row chunks."""
import pytest

from paper_2605_10380_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("min_split", ["128", "256", "384", "512"])
@pytest.mark.parametrize("q,hq,hkv", [(1, 32, 8), (2, 32, 8), (5, 24, 8), (5, 32, 8), (8, 32, 8), (3, 8, 8)])
@pytest.mark.parametrize("merge", ["1", "0"], ids=["cluster", "memory"])
def test_tiles_and_rows(q, hq, hkv, min_split, merge, monkeypatch):
    import oracle
    from tests.gpu_util import DeviceBatch, check_attention, oracle_pools_after_append
    monkeypatch.setenv("AGX_SMALL_MIN_SPLIT", min_split)
    monkeypatch.setenv("AGX_CLUSTER_MERGE", merge)
    for P in (0, 120, 121, 250, 384, 1100, 1900):
        w = W.make_attn_workload("short", P + q, "bf16", hq, hkv, 128, [P], [q], spare_pages=1)
        b = DeviceBatch(w)
        out, lse = b.attend_append()
        assert b.status() == 0
        kp, vp = oracle_pools_after_append(w)
        ref, _ = oracle.attn_paged_batch(w.q_block, kp, vp, w.page_table, w.dtype, w.prefix_len, w.q_len, w.cu_q)
        check_attention(out, ref, f"short {P}")


def test_several_row_chunks():
    import oracle
    from tests.gpu_util import DeviceBatch, check_attention, oracle_pools_after_append
    w = W.make_attn_workload("chunks", 4, "bf16", 40, 1, 128, [300], [1], spare_pages=1)
    b = DeviceBatch(w)
    out, _ = b.attend_append()
    assert b.status() == 0
    kp, vp = oracle_pools_after_append(w)
    ref, _ = oracle.attn_paged_batch(w.q_block, kp, vp, w.page_table, w.dtype, w.prefix_len, w.q_len, w.cu_q)
    check_attention(out, ref, "chunks")
