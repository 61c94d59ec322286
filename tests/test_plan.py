"""The launch planner, without a GPU: what any plan has to hold, and which kernel takes which blocks."""
import numpy as np
import pytest

from tests.plan_util import accept_chunks, plan

ROWS = {"small1": 16, "small2": 32, "small4": 64, "stream": 128, "tile": 256, "simt": 8}
UNIT = {"small1": 16, "small2": 16, "small4": 16, "stream": 128, "tile": 128, "simt": 16}


def check(P, Q, hq, hkv, d, dtype):
    """Every sequence once, its splits cover its tokens, CTAs and partial slots are dealt without gap or overlap."""
    pl = plan(P, Q, hq, hkv, d, dtype)
    assert pl.status == 0, pl.error
    G, seen, slots = hq // hkv, set(), []
    for ln in pl.launches:
        items = 0
        assert 1 <= len(ln.seqs) <= 48 and ln.rows == sum(int(Q[s.index]) for s in ln.seqs)
        for s in ln.seqs:
            p, q = int(P[s.index]), int(Q[s.index])
            assert s.index not in seen
            seen.add(s.index)
            assert s.row_chunks == -(-q * G // ROWS[ln.kind]) and s.split_tokens % UNIT[ln.kind] == 0
            assert s.nsplit * s.split_tokens >= p + q
            if ln.cluster:
                assert s.nsplit == ln.cluster <= 16
            else:
                assert (s.nsplit - 1) * s.split_tokens < p + q   # (no split without tokens)
                if s.nsplit > 1:
                    slots.append((s.part_base, q * hq * s.nsplit))
            assert s.item0 == items
            items += hkv * s.row_chunks * s.nsplit
        assert ln.items == items
        if ln.kind in ("small1", "small2"):
            assert all(s.row_chunks == 1 for s in ln.seqs)
    assert seen == set(range(len(P)))
    at = 0
    for base, n in sorted(slots):
        assert base == at
        at += n
    assert at == pl.part_entries
    return pl


@pytest.mark.parametrize("hq,hkv,d,dtype", [(32, 8, 128, "bf16"), (24, 8, 128, "bf16"), (40, 8, 128, "bf16"), (16, 2, 128, "bf16"), (8, 8, 128, "bf16"),
                                            (4, 1, 128, "bf16"), (8, 2, 64, "bf16"), (4, 2, 64, "f32"), (32, 8, 128, "f32")])
def test_any_plan_is_sound(hq, hkv, d, dtype):
    rng = np.random.default_rng(hq * 100 + hkv)
    lengths = lambda lo, hi, n: np.exp(rng.uniform(np.log(lo), np.log(hi), n)).astype(np.int64)  # noqa: E731
    for i in range(150):
        B = int(lengths(1, 130, 1)[0])
        P = lengths(1, 40000, B) - 1
        Q = lengths(1, 2500, B) if i % 3 == 0 else np.where(rng.random(B) < 0.7, rng.integers(1, 17, B), lengths(16, 1500, B)) if i % 3 == 1 else np.full(B, i % 9 + 1)
        if i % 2:
            P[:] = P[0]
        check(P, Q, hq, hkv, d, dtype)


def test_which_kernel_takes_which_rows():
    """(rows per KV head: q * hq / hkv)"""
    for rows, kind in ((16, "small1"), (17, "small2"), (32, "small2"), (33, "stream"), (384, "stream"), (385, "tile")):
        assert plan([300], [rows], 8, 8).kind_of(0) == kind
    assert plan([300], [1], 40, 1).kind_of(0) == "stream"   # 40 rows of one token
    assert plan([300], [8], d=64).kind_of(0) == "simt" and plan([300], [8], dtype="f32").kind_of(0) == "simt"


@pytest.mark.parametrize("hq,hkv,d,dtype", [(32, 8, 128, "bf16"), (4, 1, 128, "bf16"), (4, 1, 64, "f32")])
def test_lengths_beyond_what_the_planner_counts_are_refused(hq, hkv, d, dtype):
    for P, Q in ((2**31 - 8, 7), (2**31 - 48, 8), (2**31 - 1, 1), (2**31 - 1, 2**30), (2**31 - 4000, 8)):
        assert plan([100, P], [1, Q], hq, hkv, d, dtype).status == -2   # AGX_E_RANGE, no exception
    for P in (2**31 - 5000, 1500000000, 2**30):
        check([P, 100], [1, 8], hq, hkv, d, dtype)
        check([P], [8], hq, hkv, d, dtype)


def test_forced_cross_overs(monkeypatch):
    """AGX_BATCH_STREAM_TOKENS replaces the rule for batches only, AGX_STREAM_MIN_TOKENS that for one sequence only; they can be given together."""
    def kinds(P, Q):
        return [plan(P, Q).kind_of(s) for s in range(len(P))]
    monkeypatch.setenv("AGX_BATCH_STREAM_TOKENS", "20000")
    assert kinds([60000], [8]) == ["stream"] and kinds([10230], [2]) == ["small1"] == kinds([10230], [1]) and kinds([10240], [2]) == ["stream"]
    assert kinds([7100], [8]) == ["small2"] and kinds([7168], [8]) == ["stream"] and kinds([7168], [3]) == ["stream"]
    assert kinds([9000, 12000], [1, 1]) == ["stream"] * 2 and kinds([9000, 9000], [1, 1]) == ["small1"] * 2
    assert kinds([900, 12000], [1, 1]) == ["small1", "stream"]
    monkeypatch.setenv("AGX_STREAM_MIN_TOKENS", "500")
    assert kinds([400, 600], [1, 1]) == ["small1", "stream"] and kinds([400] * 51, [1] * 51) == ["stream"] * 51
    monkeypatch.delenv("AGX_BATCH_STREAM_TOKENS")
    assert kinds([400] * 51, [1] * 51) == ["small1"] * 51 and kinds([600], [1]) == ["stream"]


@pytest.mark.parametrize("P,q,items", [([2500] * 4, 1, 288), ([2500] * 6, 4, 288), ([2500] * 4, 8, 288), ([4650] * 2, 4, 288), ([6000] * 4, 4, 288),
                                       ([5102, 1819, 1520], 4, 296), ([1500] * 12, 1, 288), ([2500] * 8, 1, 256), ([300] * 32, 1, 256)])
def test_one_wave_of_small_blocks_fills_the_half_sms(P, q, items):
    """Two CTAs per SM: as many splits as are one wave, in steps of a page."""
    ln, = plan(P, [q] * len(P)).launches
    assert ln.kw == 4 and ln.items == items <= 296


def test_three_tiles_of_a_wide_block_are_not_split():
    for q, hq, hkv in ((5, 16, 2), (8, 16, 2), (8, 40, 8)):
        assert plan([300], [q], hq, hkv).launches[0].seqs[0].nsplit == 1
        assert plan([1000], [q], hq, hkv).launches[0].seqs[0].nsplit == 4


def test_chains_of_the_fp32_kernel_are_bounded():
    """Tiles of 64 tokens per CTA where a launch is a few waves; what fills the GPU unsplit stays so."""
    def longest(P, Q):
        return max(s.split_tokens for l in plan(P, Q, dtype="f32", hq=32, hkv=8).launches for s in l.seqs)
    assert longest([20000] + [40] * 30, [1] * 31) <= 256 and longest([8000] * 6, [1] * 6) <= 256 and longest([1000] * 16, [1] * 16) == 512
    assert plan([0], [4000], dtype="f32", hq=32, hkv=8).launches[0].seqs[0].nsplit == 1


@pytest.mark.parametrize("q", [3, 8])
def test_one_block_has_a_shorter_last_split(q):
    """Blocks of one sequence in splits that an SM holds whole: at most 16, the last one with a KV tile less than the others."""
    shorter = 0
    for L in range(270, 6200, 37):
        ln = plan([L - q], [q]).launches[0]
        s = ln.seqs[0]
        if ln.kind in ("small1", "small2") and s.split_tokens <= 384 and not ln.cluster and not ln.lean:
            last = L - (s.nsplit - 1) * s.split_tokens
            assert 2 <= s.nsplit <= 16 and 0 < last <= s.split_tokens
            shorter += -(-last // 128) < -(-s.split_tokens // 128)
    assert shorter > 100


@pytest.mark.parametrize("P,q,hq,hkv", [(3000, 256, 32, 8), (2364, 308, 24, 8), (875, 225, 32, 8), (1500, 200, 32, 8), (5000, 256, 16, 2)])
def test_a_few_long_splits_are_not_left_for_a_second_wave(P, q, hq, hkv):
    """A split prefill of about one wave: the CTAs with tokens fit the SMs at once, or all of them take part in the second wave."""
    ln, = plan([P], [q], hq, hkv).launches
    assert ln.kind == "tile"
    s, G, busy = ln.seqs[0], hq // hkv, 0
    for rc in range(s.row_chunks):
        seen = P + min(q - 1, (256 * rc + 255) // G) + 1
        busy += hkv * min(s.nsplit, -(-seen // s.split_tokens))
    assert busy <= 148 or busy >= 1.5 * 148


@pytest.mark.parametrize("hq,hkv", [(32, 8), (24, 8), (40, 8), (16, 2), (8, 8), (4, 1)])
def test_one_block_is_split_from_257_tokens_on(hq, hkv):
    """What one CTA holds whole in two KV tiles needs no second launch."""
    for q in range(1, 17):
        for L in range(130, 300, 3):
            ln, = plan([L - q], [q], hq, hkv).launches
            if ln.kind in ("small1", "small2"):
                assert (ln.seqs[0].nsplit > 1) == (L > 256), (L, q)


@pytest.mark.parametrize("prefix,q,hq,splits", [
    ([4000, 4000, 8000], [1000, 500, 400], 32, [1, 1, 1]),
    ([8000, 6000, 1000], [700, 400, 200], 24, [1, 1, 1]),
    ([3000, 2000, 0], [400, 400, 700], 24, [2, 2, 1]),
    ([6000, 1000, 3000, 8000, 4000], [200, 200, 700, 500, 500], 32, [1, 1, 1, 1, 1]),
    ([3178], [958], 24, [3]),                               # (one block: what it saves to split is more, 62.6 / 52.4 us a layer)
])
def test_splits_of_several_prefills(prefix, q, hq, splits):
    """Three and more blocks of the 256-row schedule keep each other's SMs busy: a merge behind them costs what it did before its costs were fitted to lone blocks."""
    ln, = plan(prefix, q, hq, 8).launches
    assert ln.kind == "tile" and [s.nsplit for s in sorted(ln.seqs, key=lambda s: s.index)] == splits


@pytest.mark.parametrize("rows,vocab,elem_bytes,aligned,chunks", [
    (64, 128256, 2, True, 13), (444, 128256, 2, True, 2), (445, 128256, 2, True, 1), (888, 128256, 2, True, 1), (64, 4096, 2, True, 1),   # one wave
    (889, 128256, 2, True, 2), (1332, 128256, 2, True, 2), (1333, 128256, 2, True, 1), (1776, 128256, 2, True, 2),                        # and the one that is left
    (889, 32000, 4, True, 2), (889, 32000, 2, True, 1),
    (445, 32003, 2, False, 3), (256, 128257, 2, False, 5), (889, 128257, 2, False, 2), (4000, 128257, 2, False, 1), (33, 2000, 2, False, 1),
])
def test_chunks_of_a_logits_row(rows, vocab, elem_bytes, aligned, chunks):
    """One wave of CTAs where rows are read 16 bytes a load, eight CTAs an SM rounded up where an element a load."""
    assert accept_chunks(rows, vocab, elem_bytes, aligned) == chunks
