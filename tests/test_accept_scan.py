"""The accept step: natural ties, special values, remainders of vectors, chunks and warps."""
import numpy as np
import pytest

from paper_2605_10380_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("vocab", [2, 7, 8, 129, 1000, 1024, 32003, 128256])
@pytest.mark.parametrize("q", [[1], [1, 3], [5, 1, 9, 2], [1] * 40], ids=["1", "4", "17", "40"])
def test_accept_against_the_oracle(dtype, vocab, q):
    import oracle
    from paper_2605_10380_b200 import agx
    from tests.gpu_util import run_accept
    stride = (vocab + 7) // 8 * 8 + 8
    P = [100 + 3 * i for i in range(len(q))]
    aw = W.make_planted_accept("acc", vocab + len(q), dtype, vocab, q, P, row_stride=stride)
    f = W.storage_to_f32(aw.logits, dtype).copy()
    rng = np.random.default_rng(vocab)
    rows = f.shape[0]
    f[0, :vocab] = np.round(f[0, :vocab])                       # many ties
    if rows > 2:
        f[1, :vocab] = np.nan                                   # nothing but NaN: token 0
        f[2, :vocab] = -np.inf
        f[2, rng.integers(0, vocab)] = np.nan
    if rows > 5:
        f[3, :vocab] = -0.0                                     # -0 and +0 tie
        f[3, vocab // 2] = 0.0
        f[4, rng.integers(0, vocab, size=3)] = np.inf
        f[5, :vocab] = -np.abs(f[5, :vocab]) - 1                # all negative
    aw.logits = W.to_storage(f, dtype)
    got = run_accept(agx.Handle(32, 8, 128, "bf16"), aw)
    ref = oracle.accept_greedy(aw.logits, dtype, aw.vocab, aw.drafts, aw.cu_q, aw.prefix_len)
    for g, r in zip(got, ref):
        assert np.array_equal(g, r)


@pytest.mark.parametrize("dtype,vocab", [("f32", 2), ("f32", 517), ("f32", 4096), ("f32", 4100), ("bf16", 8192), ("bf16", 8200), ("bf16", 60000)])
@pytest.mark.parametrize("q", [[2], [2, 1], [3, 2], [1, 1, 4], [7], [1] * 8, [8], [4, 5]], ids=["2", "3", "5", "6", "7", "8x1", "8", "9"])
def test_few_rows_on_both_sides_of_one_cluster(dtype, vocab, q):
    """Up to eight rows of at most 16 KB a CTA are one cluster's, more or longer ones are not; longest matches of drafts in both."""
    import oracle
    from paper_2605_10380_b200 import agx
    from tests.gpu_util import run_accept
    aw = W.make_planted_accept("few", vocab + sum(q), dtype, vocab, q, [50 + i for i in range(len(q))], row_stride=(vocab + 7) // 8 * 8)
    got = run_accept(agx.Handle(32, 8, 128, "bf16"), aw)
    ref = oracle.accept_greedy(aw.logits, dtype, aw.vocab, aw.drafts, aw.cu_q, aw.prefix_len)
    for g, r in zip(got, ref):
        assert np.array_equal(g, r)
