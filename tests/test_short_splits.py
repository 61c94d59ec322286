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


@pytest.mark.parametrize("q,lengths", [
    (8, [6518]), (8, [6522]), (8, [6902]), (8, [6906]), (8, [7000]),   # 17 and 18 splits of 384 tokens, and the first that need longer ones
    (1, [1000] * 6), (8, [1000] * 6), (8, [1000] * 7), (8, [3700, 3900]), (8, [1500, 2500, 3500]),   # one wave of 384 tokens or not, alike or ragged
])
def test_edge_of_whole_splits(q, lengths):
    import oracle
    from tests.gpu_util import DeviceBatch, check_attention, oracle_pools_after_append
    w = W.make_attn_workload("edge", sum(lengths) + q, "bf16", 32, 8, 128, lengths, [q] * len(lengths), spare_pages=1)
    b = DeviceBatch(w)
    out, _ = b.attend_append()
    assert b.status() == 0
    kp, vp = oracle_pools_after_append(w)
    ref, _ = oracle.attn_paged_batch(w.q_block, kp, vp, w.page_table, w.dtype, w.prefix_len, w.q_len, w.cu_q)
    check_attention(out, ref, "edge")
