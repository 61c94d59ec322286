"""Kernel for short KV splits with swapped MMA operands: 4, 8, 16 and 32 columns of query rows, one to three tiles of 128 tokens (the last
one short), splits merged through memory, in a cluster or not at all, the last blocks it takes and the first it does not.  Which kernel takes a
block is checked against the planner."""
import pytest

from paper_2605_10380_b200 import workloads as W
from tests.plan_util import plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("min_split", ["128", "256", "384", "512"])
@pytest.mark.parametrize("q,hq,hkv", [(1, 32, 8), (2, 32, 8), (5, 24, 8), (5, 32, 8), (8, 32, 8), (3, 8, 8)])
@pytest.mark.parametrize("merge", ["1", "0"], ids=["cluster", "memory"])
def test_tiles_and_rows(q, hq, hkv, min_split, merge, monkeypatch):
    import oracle
    from tests.gpu_util import DeviceBatch, check_attention, oracle_pools_after_append
    monkeypatch.setenv("AGX_SMALL_MIN_SPLIT", min_split)
    monkeypatch.setenv("AGX_CLUSTER_MERGE", merge)
    monkeypatch.setenv("AGX_STREAM_MIN_TOKENS", "100000")   # (the small-q kernels, whatever they are estimated at)
    for P in (0, 120, 121, 250, 384, 1100, 1900):
        ln, = plan([P], [q], hq, hkv).launches
        whole = ln.seqs[0].split_tokens <= 384   # (longer splits go to the warp-MMA kernel)
        assert ln.kind in ("small1", "small2") and ln.kw == 8 and whole == (min_split != "512" or P not in (384, 1900))
        w = W.make_attn_workload("short", P + q, "bf16", hq, hkv, 128, [P], [q], spare_pages=1)
        b = DeviceBatch(w)
        out, lse = b.attend_append()
        assert b.status() == 0
        kp, vp = oracle_pools_after_append(w)
        ref, _ = oracle.attn_paged_batch(w.q_block, kp, vp, w.page_table, w.dtype, w.prefix_len, w.q_len, w.cu_q)
        check_attention(out, ref, f"short {P}")


@pytest.mark.parametrize("q,hq,hkv,kind", [(16, 8, 8, "small1"), (17, 8, 8, "small2"), (32, 8, 8, "small2"), (33, 8, 8, "stream"),
                                           (1, 16, 1, "small1"), (1, 32, 1, "small2"), (1, 40, 1, "stream")])
def test_edges_of_the_rows(q, hq, hkv, kind):
    """16, 17, 32 and 33 rows per KV head, of many tokens or of one."""
    import oracle
    from tests.gpu_util import DeviceBatch, check_attention, oracle_pools_after_append
    ln, = plan([300], [q], hq, hkv).launches
    assert ln.kind == kind and (kind == "stream" or ln.seqs[0].split_tokens <= 384)
    w = W.make_attn_workload("rows", 4 + q, "bf16", hq, hkv, 128, [300], [q], spare_pages=1)
    b = DeviceBatch(w)
    out, _ = b.attend_append()
    assert b.status() == 0
    kp, vp = oracle_pools_after_append(w)
    ref, _ = oracle.attn_paged_batch(w.q_block, kp, vp, w.page_table, w.dtype, w.prefix_len, w.q_len, w.cu_q)
    check_attention(out, ref, "rows")


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
