"""Warp-MMA kernel with two tiles per warp: splits of one, two and three ring stages are taken in pairs of stages, longer ones stage by
stage; the last stage of each may be short."""
import pytest

from paper_2605_10380_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("min_split", ["128", "256", "384", "512", "2048"])
@pytest.mark.parametrize("q", [5, 8])
def test_stages_per_trip(q, min_split, monkeypatch):
    import oracle
    from tests.gpu_util import DeviceBatch, check_attention, oracle_pools_after_append
    monkeypatch.setenv("AGX_SMALL_MIN_SPLIT", min_split)
    for P in (120, 121, 129, 250, 384, 512, 1100, 1900):
        w = W.make_attn_workload("pairs", P + q, "bf16", 32, 8, 128, [P], [q], spare_pages=1)
        b = DeviceBatch(w)
        out, _ = b.attend_append()
        assert b.status() == 0
        kp, vp = oracle_pools_after_append(w)
        ref, _ = oracle.attn_paged_batch(w.q_block, kp, vp, w.page_table, w.dtype, w.prefix_len, w.q_len, w.cu_q)
        check_attention(out, ref, f"pairs {P}")
