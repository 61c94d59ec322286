"""The accept step where the number of chunks a row is cut into changes: as many rows as CTAs of a wave, half of them, one more; chunks whose threads
have one to eight vectors, with a vector cut by the end of the row."""
import numpy as np
import pytest

from paper_2605_10380_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,vocab", [("bf16", 4103), ("bf16", 20011), ("bf16", 66000), ("f32", 9001), ("f32", 32003)])
@pytest.mark.parametrize("rows", [17, 100, 444, 445, 888, 889])
def test_rows_and_chunks(dtype, vocab, rows):
    import oracle
    from paper_2605_10380_b200 import agx
    from tests.gpu_util import run_accept
    q = [4] * (rows // 4) + ([rows % 4] if rows % 4 else [])
    aw = W.make_planted_accept("chunks", vocab + rows, dtype, vocab, q, [60 + i % 9 for i in range(len(q))], row_stride=(vocab + 7) // 8 * 8)
    f = W.storage_to_f32(aw.logits, dtype).copy()
    f[::3, vocab - 1] = 9.0                     # winners in the cut vector and, tied with it, at the start
    f[::6, 0] = 9.0
    aw.logits = W.to_storage(f, dtype)
    got = run_accept(agx.Handle(32, 8, 128, "bf16"), aw)
    ref = oracle.accept_greedy(aw.logits, dtype, aw.vocab, aw.drafts, aw.cu_q, aw.prefix_len)
    for g, r in zip(got, ref):
        assert np.array_equal(g, r)


@pytest.mark.parametrize("dtype,vocab,stride", [("bf16", 32003, 32003), ("bf16", 9001, 9003), ("f32", 8005, 8005)])
@pytest.mark.parametrize("rows", [17, 256, 445, 889])
def test_rows_off_16_bytes(dtype, vocab, stride, rows):
    """Rows that do not start on 16 bytes: an element a load, chunks by a rule of their own."""
    import oracle
    from paper_2605_10380_b200 import agx
    from tests.gpu_util import run_accept
    q = [4] * (rows // 4) + ([rows % 4] if rows % 4 else [])
    aw = W.make_planted_accept("off", vocab + rows, dtype, vocab, q, [60 + i % 9 for i in range(len(q))], row_stride=stride)
    f = W.storage_to_f32(aw.logits, dtype).copy()
    f[::3, vocab - 1] = 9.0
    f[::6, 0] = 9.0
    aw.logits = W.to_storage(f, dtype)
    got = run_accept(agx.Handle(32, 8, 128, "bf16"), aw)
    ref = oracle.accept_greedy(aw.logits, dtype, aw.vocab, aw.drafts, aw.cu_q, aw.prefix_len)
    for g, r in zip(got, ref):
        assert np.array_equal(g, r)
