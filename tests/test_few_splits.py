"""Merge of the partials of two to eight KV splits: fp16 rows in tiles (256-row schedule; row groups of whole and of cut tiles, a batch of sequences with
different and with no splits), a half-warp a (row, head) pair, and fp32 rows in slots, odd numbers of pairs; and the swapped-operand kernel with two threads
a token, at the row counts where its halves begin and end."""
import numpy as np
import pytest

from paper_2605_10380_b200 import workloads as W
from tests.plan_util import plan

pytestmark = pytest.mark.gpu


def check(prefix, q, hq, hkv, what):
    import oracle
    from tests.gpu_util import DeviceBatch, check_attention, oracle_pools_after_append
    w = W.make_attn_workload(what, sum(prefix) + sum(q), "bf16", hq, hkv, 128, prefix, q, spare_pages=1)
    b = DeviceBatch(w)
    out, lse = b.attend_append()
    assert b.status() == 0
    again, _ = b.attend_append()
    assert (again == out).all()   # splits are added in order
    kp, vp = oracle_pools_after_append(w)
    ref, ref_lse = oracle.attn_paged_batch(w.q_block, kp, vp, w.page_table, w.dtype, w.prefix_len, w.q_len, w.cu_q)
    check_attention(out, ref, what)
    # (fp32 results of 2 to 9, half an ulp 2^-22, behind scores of exact products, sums and logarithms in fp32: at most 1.1e-6 measured over all of these shapes)
    assert np.abs(lse - ref_lse).max() <= 5e-6


@pytest.mark.parametrize("splits", [2, 3, 4, 5, 7, 8])
@pytest.mark.parametrize("q,hq,hkv", [(129, 8, 2), (131, 3, 1), (400, 1, 1)])
def test_partials_in_tiles(q, hq, hkv, splits, monkeypatch):
    monkeypatch.setenv("AGX_TILE_SPLIT_TOKENS", "128")
    monkeypatch.setenv("AGX_STREAM_MAX_ROWS", "32")   # (the 256-row schedule, whatever it is estimated at)
    P = max(0, 128 * splits - 37 - q)
    ln, = plan([P], [q], hq, hkv).launches
    assert ln.kind == "tile" and ln.seqs[0].nsplit == max(splits, (P + q + 127) // 128)
    check([P], [q], hq, hkv, f"tiles {splits}")


def test_partials_in_tiles_of_a_batch(monkeypatch):
    monkeypatch.setenv("AGX_TILE_SPLIT_TOKENS", "256")
    monkeypatch.setenv("AGX_STREAM_MAX_ROWS", "32")
    prefix, q = [700, 0, 30, 1500], [90, 200, 85, 257]
    ln, = plan(prefix, q, 6, 2).launches
    assert sorted(s.nsplit for s in ln.seqs) == [1, 1, 4, 7]
    check(prefix, q, 6, 2, "batch")


@pytest.mark.parametrize("n,tokens,q,hq,hkv,kind,splits", [
    (6, 800, 1, 32, 8, "small1", 3), (3, 1500, 3, 32, 8, "small1", 5), (3, 1500, 1, 32, 8, "small1", 6), (2, 2000, 8, 24, 8, "small2", 8),
    (1, 500, 8, 16, 2, "stream", 2), (1, 500, 16, 24, 8, "stream", 3), (1, 800, 8, 16, 2, "stream", 4), (1, 2000, 8, 16, 2, "stream", 8),
])
def test_partials_in_slots(n, tokens, q, hq, hkv, kind, splits):
    ln, = plan([tokens] * n, [q] * n, hq, hkv).launches
    assert ln.lean and ln.kind == kind and ln.seqs[0].nsplit == splits
    check([tokens] * n, [q] * n, hq, hkv, "slots")


@pytest.mark.parametrize("rows", [5, 8, 9, 12, 13, 16, 17, 20, 24, 25, 31, 32])
@pytest.mark.parametrize("tokens", [40, 129, 250, 300, 511])
def test_two_threads_a_token(rows, tokens):
    """Rows of one head a group, so that any number of them may be there."""
    ln, = plan([tokens], [rows], 2, 2).launches
    assert ln.kind in ("small1", "small2") and ln.kw == 8 and ln.seqs[0].split_tokens <= 256 and not ln.cluster
    check([tokens], [rows], 2, 2, f"{rows} rows")


@pytest.mark.parametrize("q,G", [(3, 3), (4, 3), (5, 3), (7, 3), (10, 3), (3, 4), (4, 4), (5, 4), (6, 4), (8, 4)])
@pytest.mark.parametrize("tokens", [29, 127, 128, 252, 255, 300, 511])
def test_two_threads_a_token_of_a_group(q, G, tokens):
    """Several heads a group: a token's rows lie on both sides of the halves, and so does the edge up to which the block's rows see."""
    ln, = plan([tokens], [q], 2 * G, 2).launches
    assert ln.kind in ("small1", "small2") and ln.kw == 8 and ln.seqs[0].split_tokens <= 256 and not ln.cluster
    check([tokens], [q], 2 * G, 2, f"{q} x {G} rows")
