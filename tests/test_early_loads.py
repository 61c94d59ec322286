"""Early loads of cached-prefix pages where the block's own pages come from the pool too, written by the launch directly in front, with
whatever the pool held behind the last token."""
import pytest

from paper_2605_10380_b200 import workloads as W

pytestmark = pytest.mark.gpu

CASES = {
    # name: (prefix lengths, q, heads, environment)
    "short_splits": ([300, 16, 1, 1900], 8, (32, 8), {}),
    "warp_mma_4_page_stages": ([1000, 500, 2044, 15], 4, (32, 8), {"AGX_SMALL_KW": "4", "AGX_SMALL_MIN_SPLIT": "1024"}),
    "warp_mma_8_page_stages": ([1000, 500, 2044, 15], 8, (32, 8), {"AGX_SMALL_KW": "8", "AGX_SMALL_MIN_SPLIT": "1024", "AGX_STREAM_MIN_TOKENS": "100000"}),
    "page_ids_over_two_groups": ([500, 1020], 30, (8, 8), {"AGX_SMALL_KW": "4", "AGX_SMALL_MIN_SPLIT": "2048"}),
    "64_rows": ([400, 1015], 16, (32, 8), {"AGX_FORCE_MMA_SYNC": "1"}),
    "row_chunks_more_pages_than_stages": ([400, 37], 600, (4, 4), {"AGX_FORCE_MMA_SYNC": "1", "AGX_SMALL_MIN_SPLIT": "2048"}),
}


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("shift", [0, 1, 9, 15])
def test_block_pages_follow_the_wait(case, shift, monkeypatch):
    import torch

    from paper_2605_10380_b200 import agx
    from tests.gpu_util import DeviceBatch
    prefixes, q, (hq, hkv), env = CASES[case]
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    P = [p + shift for p in prefixes]
    w = W.make_attn_workload("early", sum(P), "bf16", hq, hkv, 128, P, [q] * len(P), spare_pages=1)
    outs = {}
    for early in (0, 1):
        b = DeviceBatch(w)
        for s, p in enumerate(P):   # the pool behind the last token
            if (p + q) % 16:
                for pool in (b.k_pool, b.v_pool):
                    pool[int(w.page_table[s, (p + q) // 16]), :, (p + q) % 16:] = float("nan")
        b.h.set_option(agx.AGX_OPT_EARLY_PREFIX_LOADS, early)
        gen = torch.Generator(device="cuda")
        gen.manual_seed(3)
        rows = [[torch.randn(b.k_new.shape, generator=gen, device="cuda").to(torch.bfloat16) for _ in range(2)] for _ in range(8)]
        outs[early] = [torch.zeros_like(b.out) for _ in rows]
        torch.cuda.synchronize()
        for (k, v), out in zip(rows, outs[early]):   # nothing but the library's launches, one right behind the other
            b.h.kv_append(b.k_pool, b.v_pool, k, v, b.page_table, b.prefix_len, b.cu_q)
            b.h.attn_prefixed(b.q_block, b.k_pool, b.v_pool, b.page_table, w.prefix_len, w.q_len, out, None, b.ws)
        torch.cuda.synchronize()
        assert b.status() == 0
    for a, c in zip(outs[0], outs[1]):
        assert bool(torch.isfinite(a.float()).all()) and torch.equal(a, c)
