"""Values far from 1: split partials of the 256-row schedule are fp16 rows, and whatever magnitude V has must come through them as it does through the fp32
rows of the other kernels.  Each kernel that leaves partials with each merge that reads them, V scaled by powers of two: all of it, differently by column, by
token (so that the splits of a row differ), every other KV head, and with an infinite value in it."""
import numpy as np
import pytest

from paper_2605_10380_b200 import workloads as W
from tests.plan_util import plan

pytestmark = pytest.mark.gpu

WIDE = {"AGX_STREAM_MAX_ROWS": "32"}   # (more than 32 rows: the 256-row schedule, whatever it is estimated at)
T128 = {**WIDE, "AGX_TILE_SPLIT_TOKENS": "128"}
LONG = {"AGX_SMALL_MIN_SPLIT": "512", "AGX_CLUSTER_MERGE": "0"}   # (splits that no SM holds whole: 8-page stages)
# environment, sequences, tokens in front, rows, query heads, KV heads -> kernel, splits
SHAPES = [
    (T128, 1, 218, 129, 8, 2, "tile", 3), (T128, 1, 730, 129, 8, 2, "tile", 7), (T128, 1, 1370, 129, 8, 2, "tile", 12), (T128, 1, 4058, 129, 8, 2, "tile", 33),
    ({}, 1, 0, 897, 24, 8, "tile", 2),
    ({}, 6, 800, 1, 32, 8, "small1", 3), ({}, 3, 1500, 3, 32, 8, "small1", 5), ({}, 2, 2000, 8, 24, 8, "small2", 8), ({}, 1, 9000, 8, 8, 2, "small2", 36),
    (LONG, 1, 3000, 3, 8, 2, "small1", 6), (LONG, 1, 3000, 8, 8, 2, "small2", 6), ({**WIDE, "AGX_CLUSTER_MERGE": "0"}, 1, 900, 12, 8, 2, "small4", 4),
    ({}, 1, 500, 8, 16, 2, "stream", 2), ({}, 1, 2000, 8, 16, 2, "stream", 8), ({}, 1, 6000, 8, 16, 2, "stream", 24),
]


def scales(what, tokens):
    """Powers of two by which V is scaled: [tokens][128]."""
    tok, col = np.arange(tokens)[:, None], np.arange(128)[None, :]
    e = {"tiny": -20, "huge": 20, "least": -100, "most": 100, "infinite": 24, "heads": 0, "columns": 4 * (col // 16) - 60, "tokens": 20 * (tok // 64 % 3) - 24}[what]
    return np.exp2(np.broadcast_to(np.asarray(e, np.float32), (tokens, 128)))


@pytest.mark.parametrize("what", ["tiny", "huge", "least", "most", "columns", "tokens", "heads", "infinite"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: f"{s[6]}-{s[7]}")
def test_any_magnitude(shape, what, monkeypatch):
    import oracle
    from tests.gpu_util import RTOL, DeviceBatch, oracle_pools_after_append
    env, n, P, q, hq, hkv, kind, splits = shape
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    ln, = plan([P] * n, [q] * n, hq, hkv).launches
    assert ln.kind == kind and ln.seqs[0].nsplit == splits and not ln.cluster
    w = W.make_attn_workload("range", P + q, "bf16", hq, hkv, 128, [P] * n, [q] * n, spare_pages=1)
    f = scales(what, P + q)
    page, new = W.storage_to_f32(w.v_pool, "bf16").copy(), W.storage_to_f32(w.v_new, "bf16").copy()   # [pages][hkv][16][128], [rows][hkv][128]
    for s in range(n):
        for t in range(0, P + q, 16):
            ids, k = w.page_table[s, t // 16], min(16, P + q - t)
            page[ids, :, :k] *= f[t:t + k]
        new[s * q:(s + 1) * q] *= f[P:, None]
        if what == "infinite":   # (column 37 of the first token, which every row sees)
            page[w.page_table[s, 0], :, 0, 37] = np.inf
            if P == 0:
                new[s * q, :, 37] = np.inf
    if what == "heads":
        page[:, 1::2] *= 2.0 ** -30
        new[:, 1::2] *= 2.0 ** -30
    w.v_pool, w.v_new = W.to_storage(page, "bf16"), W.to_storage(new, "bf16")
    b = DeviceBatch(w)
    out, lse = b.attend_append()
    assert b.status() == 0
    kp, vp = oracle_pools_after_append(w)
    ref, ref_lse = oracle.attn_paged_batch(w.q_block, kp, vp, w.page_table, w.dtype, w.prefix_len, w.q_len, w.cu_q)
    if what == "infinite":
        assert not np.isfinite(out[..., 37]).any()
        out[..., 37] = ref[..., 37] = 0
    # the usual bound on a row's error against its largest value, for every 16 columns by themselves (they differ in magnitude under "columns")
    out, ref = out.reshape(-1, 8, 16), ref.reshape(-1, 8, 16)
    assert np.isfinite(out).all() and np.isfinite(ref).all()
    assert (np.abs(out - ref).max(-1) <= RTOL * np.abs(ref).max(-1)).all(), np.max(np.abs(out - ref).max(-1) / np.abs(ref).max(-1))
    assert np.abs(lse - ref_lse).max() <= 5e-6   # (V is not in it: as in test_few_splits.py)
