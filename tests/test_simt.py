"""The fp32-arithmetic attention kernel (fp32 pools, bf16 pools with head_dim 64): tile edges, row-chunk remainders, clusters of KV
splits and partials, with and without the fused append."""
import numpy as np
import pytest

from paper_2605_10380_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("merge", ["clusters", "partials"])
@pytest.mark.parametrize("dtype,d,hq,hkv", [("f32", 64, 4, 2), ("f32", 128, 8, 2), ("f32", 64, 3, 3), ("bf16", 64, 10, 2)])
def test_simt_kernel_against_the_oracle(dtype, d, hq, hkv, merge, monkeypatch):
    import torch

    import oracle
    from tests.gpu_util import DeviceBatch, check_attention, oracle_pools_after_append
    if merge == "partials":
        monkeypatch.setenv("AGX_CLUSTER_MERGE", "0")
    for P, q in (([0], [1]), ([63], [1]), ([64], [2]), ([256], [4]), ([1000, 17, 1, 500], [3, 8, 70, 1]), ([1025], [9])):
        w = W.make_attn_workload("simt", 7 * sum(P) + sum(q), dtype, hq, hkv, d, P, q, spare_pages=2)
        two = DeviceBatch(w)
        two.append()
        out, lse = two.attend()
        one = DeviceBatch(w)
        one.attend_append()
        assert one.status() == 0 and two.status() == 0
        assert torch.equal(one.k_pool, two.k_pool) and torch.equal(one.v_pool, two.v_pool)
        assert torch.equal(one.out, two.out) and torch.equal(one.lse, two.lse), (P, q)
        kp, vp = oracle_pools_after_append(w)
        ref, ref_lse = oracle.attn_paged_batch(w.q_block, kp, vp, w.page_table, w.dtype, w.prefix_len, w.q_len, w.cu_q)
        check_attention(out, ref, f"simt {P} {q}")
        # fp32 scores of d products are off by at most d 2^-24 sum |q k| / sqrt(d) ~ 5e-5; exponentials and sums add a few 1e-7
        assert np.max(np.abs(lse - ref_lse)) < 1e-4
        if dtype == "f32":
            assert np.max(np.abs(out - ref)) < 2e-4, (P, q)   # (2 x 5e-5 x max |v|)


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("dtype,d", [("f32", 64), ("f32", 128), ("bf16", 64)])
def test_what_a_row_does_not_see_does_not_reach_it(dtype, d, value):
    """V of the block's last token: earlier rows keep every bit, whichever tile and split the token sits in."""
    import torch

    from tests.gpu_util import DeviceBatch
    for P, q in ((0, 9), (60, 5), (64, 3), (1000, 12), (2500, 2)):
        outs = []
        for x in (1.0, value):
            b = DeviceBatch(W.make_attn_workload("hidden", P + q, dtype, 8, 2, d, [P], [q], spare_pages=1))
            b.v_new[q - 1] = x
            b.attend_append()
            assert b.status() == 0
            outs.append((b.out, b.lse))
        assert bool(torch.isfinite(outs[1][0][:q - 1]).all()), (P, q)
        assert torch.equal(outs[0][0][:q - 1], outs[1][0][:q - 1]) and torch.equal(outs[0][1], outs[1][1])
        assert not bool(torch.isfinite(outs[1][0][q - 1]).any())


def test_rows_of_very_many_heads():
    """65793 query heads over one KV head: the last row of the first token is the first where row * ceil(2^32 / heads) >> 32 is one too many."""
    import torch

    from tests.gpu_util import DeviceBatch
    heads, P, q = 65793, 20, 3
    assert ((heads - 1) * -(-2 ** 32 // heads)) >> 32 == 1
    b = DeviceBatch(W.make_attn_workload("heads", 11, "f32", heads, 1, 64, [P], [q], spare_pages=1))
    out, lse = (torch.from_numpy(a).cuda() for a in b.attend_append())
    assert b.status() == 0
    table = b.page_table[0].long()
    k, v = (pool[table][:, 0].reshape(-1, 64)[:P + q].double() for pool in (b.k_pool, b.v_pool))   # (with the block's rows)
    s = b.q_block.double() @ k.T / 8
    hidden = torch.arange(P + q, device="cuda")[None, :] > P + torch.arange(q, device="cuda")[:, None]
    s = s.masked_fill(hidden[:, None, :], float("-inf"))
    # (the bounds of test_simt_kernel_against_the_oracle)
    assert float((torch.softmax(s, -1) @ v - out).abs().max()) < 2e-4
    assert float((torch.logsumexp(s, -1) - lse).abs().max()) < 1e-4
