"""Blocks of 18 to 32 rows with one query head per KV head, whose rows lie in three pages of a KV split that an SM holds whole: every row goes to
the page that the page table gives it."""
import dataclasses

import numpy as np
import pytest

from paper_2605_10380_b200 import workloads as W
from tests.plan_util import plan

PREFIX = {8: 3103, 16: 2095, 32: 1440}   # splits of three KV tiles, by the number of heads
BLOCKS = [18, 24, 31, 32]


def test_their_splits_are_longer_than_two_tiles():
    for heads, P in PREFIX.items():
        for q in BLOCKS:
            n = 0
            for shift in range(16):
                ln, = plan([P + shift], [q], heads, heads).launches
                s, = ln.seqs
                assert ln.kind == "small2" and ln.kw == 8 and s.nsplit > 1
                n += 256 < s.split_tokens <= 384
            assert n == 16, (heads, q, n)


@pytest.mark.gpu
@pytest.mark.parametrize("heads", PREFIX)
@pytest.mark.parametrize("q", BLOCKS)
def test_pools_are_those_of_the_append_kernel(heads, q):
    import torch

    from tests.gpu_util import DeviceBatch
    P = PREFIX[heads]
    w = W.make_attn_workload("own", heads + q, "bf16", heads, heads, 128, [P + 15], [q], spare_pages=2)
    for shift in range(16):
        v = dataclasses.replace(w, prefix_len=np.asarray([P + shift], np.int32))
        one, two = DeviceBatch(v), DeviceBatch(v)
        one.attend_append()
        two.append()
        two.attend()
        assert one.status() == 0 and two.status() == 0
        assert torch.equal(one.k_pool, two.k_pool) and torch.equal(one.v_pool, two.v_pool), shift
        assert torch.equal(one.out, two.out) and torch.equal(one.lse, two.lse), shift
