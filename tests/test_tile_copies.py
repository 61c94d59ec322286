"""What the tensor-core schedules move by TMA: Q tiles whose rows start and end inside a token's group of heads, the block's own rows from
the tiles into the pool, and split partials in tiles of their own.  Pools bit for bit against the append kernel, everywhere; results against the
oracle with the bounds of the other parity tests."""
import pytest

from paper_2605_10380_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split_tokens", ["0", "128", "384"])
@pytest.mark.parametrize("hq,hkv,P,Q", [
    (8, 8, [0, 131, 509], [400, 523, 260]),      # one head a group: a chunk's 256 tokens lie in up to three K tiles
    (24, 8, [0, 77, 640], [257, 86, 171]),
    (40, 8, [3, 200], [300, 78]),
    (14, 2, [1000, 15], [129, 150]),
    (16, 2, [5, 250], [100, 33]),
    (66, 1, [40, 130], [20, 3]),                  # no box that fits from any row on: every row by itself
    (130, 1, [31], [7]),                          # no whole token fits a tile
    (50, 1, [17, 300], [11, 4]),                  # boxes of one token
], ids=["g1", "g3", "g5", "g7", "g8", "g66", "g130", "g50"])
def test_rows_that_do_not_meet_tiles(hq, hkv, P, Q, split_tokens, monkeypatch):
    import oracle
    import torch

    from tests.gpu_util import DeviceBatch, check_attention, oracle_pools_after_append
    monkeypatch.setenv("AGX_TILE_SPLIT_TOKENS", split_tokens)
    w = W.make_attn_workload("copies", hq + sum(P) + sum(Q), "bf16", hq, hkv, 128, P, Q, spare_pages=3)
    one, two = DeviceBatch(w), DeviceBatch(w)
    out, _ = one.attend_append()
    two.append()
    two.attend()
    assert one.status() == 0 and two.status() == 0
    assert torch.equal(one.k_pool, two.k_pool) and torch.equal(one.v_pool, two.v_pool)
    assert torch.equal(one.out, two.out)
    kp, vp = oracle_pools_after_append(w)
    ref, _ = oracle.attn_paged_batch(w.q_block, kp, vp, w.page_table, w.dtype, w.prefix_len, w.q_len, w.cu_q)
    check_attention(out, ref, "copies")


@pytest.mark.parametrize("hq,hkv,P,Q", [
    (8, 8, [0, 5, 100, 250, 1000, 127], [33, 128, 64, 129, 200, 384]),   # one Q tile, up to 128 tokens a chunk, in two tiles
    (4, 4, [1, 127, 300, 1016, 64], [385, 700, 513, 640, 400]),          # two Q tiles, 256 tokens a chunk, in three tiles: K has two stages
    (16, 8, [0, 9, 121, 640], [40, 64, 192, 100]),
    (24, 8, [3, 60, 299], [37, 120, 128]),
], ids=["stream_g1", "tile_g1", "stream_g2", "stream_g3"])
@pytest.mark.parametrize("shift", [0, 3, 8])
@pytest.mark.parametrize("split_tokens", ["0", "256"])
def test_chunks_of_many_block_rows(hq, hkv, P, Q, shift, split_tokens, monkeypatch):
    """Every whole group of eight rows leaves for the pool from the tile it is in, also where the tile's stage is filled again."""
    import torch

    from tests.gpu_util import DeviceBatch
    monkeypatch.setenv("AGX_TILE_SPLIT_TOKENS", split_tokens)
    w = W.make_attn_workload("rows", hq + sum(Q) + shift, "bf16", hq, hkv, 128, [p + shift for p in P], Q, spare_pages=3)
    one, two = DeviceBatch(w), DeviceBatch(w)
    one.attend_append()
    two.append()
    two.attend()
    assert one.status() == 0 and two.status() == 0
    assert torch.equal(one.k_pool, two.k_pool) and torch.equal(one.v_pool, two.v_pool)
    assert torch.equal(one.out, two.out) and torch.equal(one.lse, two.lse)
