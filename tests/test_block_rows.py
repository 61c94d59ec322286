"""The block's own K/V rows on their way into the attention kernels (agx_attn_prefixed_append): row groups that mix prefix and
block, whole row groups, the ragged end, at every alignment, in every schedule."""
import numpy as np
import pytest

from paper_2605_10380_b200 import workloads as W

pytestmark = pytest.mark.gpu

SCHEDULES = {
    # name: (prefix lengths around, block lengths, heads, environment)
    "warp_mma": ([0, 240, 1000], [1, 3, 8], (32, 8), {}),
    "warp_mma_two_tiles_g1": ([100, 500], [9, 31, 32], (8, 8), {}),
    "warp_mma_late_stage": ([1000, 2000], [1, 5, 8], (32, 8), {"AGX_SMALL_KW": "4", "AGX_CLUSTER_MERGE": "0", "AGX_SMALL_MIN_SPLIT": "1024"}),
    "stream": ([120, 1016], [1, 8, 17, 60], (32, 8), {"AGX_STREAM_MIN_TOKENS": "0"}),
    "tile": ([0, 120, 896], [128, 135, 300], (32, 8), {}),
    "tile_g3": ([250], [256, 333], (24, 8), {}),
}


@pytest.mark.parametrize("schedule", SCHEDULES)
@pytest.mark.parametrize("shift", [0, 1, 7, 8, 9, 15])
def test_block_rows_at_every_alignment(schedule, shift, monkeypatch):
    import torch

    from tests.gpu_util import DeviceBatch
    prefixes, blocks, (hq, hkv), env = SCHEDULES[schedule]
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    for P in prefixes:
        for q in blocks:
            # a second sequence whose block is full of NaN follows in the rows: it must not reach the first one's result
            w = W.make_attn_workload("rows", 10 * P + q + shift, "bf16", hq, hkv, 128, [P + shift, 37], [q, 5], spare_pages=1)
            two = DeviceBatch(w)
            one = DeviceBatch(w)
            for b in (two, one):
                b.k_new[q:] = float("nan")
                b.v_new[q:] = float("nan")
            # what lies in the pages from the prefix on is not read before it is written
            last = int(w.page_table[0, (P + shift) // 16])
            for pool in (one.k_pool, one.v_pool):
                pool[last, :, (P + shift) % 16:] = float("nan")
                for j in range((P + shift) // 16 + 1, (P + shift + q + 15) // 16):
                    pool[int(w.page_table[0, j])] = float("nan")
            two.append()
            two.attend()
            one.attend_append()
            assert one.status() == 0 and two.status() == 0
            assert bool(torch.isfinite(two.out[:q].float()).all())
            assert torch.equal(one.out[:q], two.out[:q]) and torch.equal(one.lse[:q], two.lse[:q]), (P, q)
            for pool, ref in ((one.k_pool, two.k_pool), (one.v_pool, two.v_pool)):
                for j in range((P + shift + q + 15) // 16):
                    n = min(16, P + shift + q - 16 * j)
                    page = int(w.page_table[0, j])
                    assert torch.equal(pool[page, :, :n], ref[page, :, :n]), (P, q, j)
            assert np.isnan(one.out[q:].float().cpu().numpy()).any()   # (the planted NaN did arrive where it belongs)
