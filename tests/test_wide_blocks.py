"""One block of 65 to 384 rows per KV head in the 256-row tensor-core schedule, with fp32 split partials in tiles."""
import pytest

from paper_2605_10380_b200 import workloads as W
from tests.plan_util import plan

# rows 65 .. 384, around the edges of warps, 128-row Q tiles and 256-row chunks; 1, 2 to 4, up to 16, up to 32 and more splits
BLOCKS = [(32, 8, 600, 64), (24, 8, 1000, 42), (40, 8, 700, 13), (32, 8, 1000, 24), (32, 8, 1000, 25), (24, 8, 2000, 43), (16, 2, 3000, 32), (32, 8, 2500, 60),
          (16, 2, 2990, 33), (66, 1, 5000, 3), (24, 8, 1000, 128), (24, 8, 0, 128), (8, 1, 5200, 17), (8, 1, 3800, 20)]


def test_schedule_of_one_block():
    for hq, hkv, P, q in BLOCKS:
        ln, = plan([P], [q], hq, hkv).launches
        assert ln.kind == "tile", (hq, hkv, P, q)
    for hq, hkv, P, q in ((32, 8, 600, 16), (8, 8, 600, 65), (32, 8, 60000, 96)):
        assert plan([P], [q], hq, hkv).kind_of(0) == "stream"
    assert plan([600, 600], [64, 64], 32, 8).kind_of(0) == "stream"


@pytest.mark.gpu
@pytest.mark.parametrize("split_tokens", ["0", "128", "384"])
@pytest.mark.parametrize("hq,hkv,P,q", BLOCKS)
def test_against_the_oracle(hq, hkv, P, q, split_tokens, monkeypatch):
    import oracle
    import torch

    from tests.gpu_util import DeviceBatch, check_attention, oracle_pools_after_append
    monkeypatch.setenv("AGX_TILE_SPLIT_TOKENS", split_tokens)
    w = W.make_attn_workload("wide", hq + P + q, "bf16", hq, hkv, 128, [P], [q], spare_pages=3)
    one, two = DeviceBatch(w), DeviceBatch(w)
    out, _ = one.attend_append()
    two.append()
    two.attend()
    assert one.status() == 0 and two.status() == 0
    assert torch.equal(one.k_pool, two.k_pool) and torch.equal(one.v_pool, two.v_pool)
    assert torch.equal(one.out, two.out) and torch.equal(one.lse, two.lse)
    kp, vp = oracle_pools_after_append(w)
    ref, _ = oracle.attn_paged_batch(w.q_block, kp, vp, w.page_table, w.dtype, w.prefix_len, w.q_len, w.cu_q)
    check_attention(out, ref, "wide")
