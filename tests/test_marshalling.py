"""The compiled argument marshalling without a GPU: what each form of an argument becomes, seen by functions that stand in for the library's."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2605_10380_b200 import agx

_FUNCTIONS = ("agx_kv_append", "agx_attn_prefixed", "agx_attn_prefixed_append", "agx_accept_greedy", "agx_verify_step_host",
              "agx_verify_step_host_enqueue", "agx_ngram_build", "agx_ngram_draft", "agx_kv_copy_pages")


@pytest.fixture
def calls():
    """(module, list of (name, arguments) of the calls made through it)"""
    lib, native, seen, keep = agx.load(), agx._binding(), [], []
    for name in _FUNCTIONS:
        def record(*args, name=name):
            seen.append((name, args))
            return 0
        keep.append(ctypes.CFUNCTYPE(ctypes.c_int32, *getattr(lib, name).argtypes)(record))
    native.bind(agx._h_i32, *(ctypes.cast(f, ctypes.c_void_p).value for f in keep))
    yield native, seen
    agx._native = None
    agx._binding()   # (one module per process: back to the library's functions)


def _tensors():
    return dict(q=torch.zeros(3, 4, 8), k=torch.zeros(3, 2, 8), v=torch.zeros(3, 2, 8), kp=torch.zeros(5, 2, 16, 8), vp=torch.zeros(5, 2, 16, 8),
                table=torch.zeros(2, 7, dtype=torch.int32), out=torch.zeros(3, 4, 8), ws=torch.zeros(100))


def test_a_copy_on_write_tensor_is_copied_before_its_address_is_taken(calls):
    native, seen = calls
    t = _tensors()
    original = torch.ones(3, 4, 8)
    lazy = torch._lazy_clone(original)
    native.attn(0, t["q"], None, None, t["kp"], t["vp"], t["table"], [1, 2], [1, 2], lazy, None, t["ws"], 0)
    out = seen[0][1][10]
    assert out == lazy.data_ptr() and out != original.data_ptr()
