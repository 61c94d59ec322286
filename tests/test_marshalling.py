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
    native.bind(agx._h_i32, np.ndarray, *(ctypes.cast(f, ctypes.c_void_p).value for f in keep))
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


class _Wrapped:
    """Not a tensor, but asked like one (a library's own array type)."""

    def __init__(self, t):
        self._t, self.shape = t, tuple(t.shape)

    def data_ptr(self):
        return self._t.data_ptr()

    def numel(self):
        return self._t.numel()

    def element_size(self):
        return self._t.element_size()

    def stride(self, i):
        return self._t.stride(i)


@pytest.mark.parametrize("wrap", [lambda t: t, _Wrapped, torch.nn.Parameter, lambda t: t.as_subclass(type("Sub", (torch.Tensor,), {}))],
                         ids=["tensor", "wrapped", "parameter", "subclass"])
def test_everything_that_is_asked_like_a_tensor_is_one(calls, wrap):
    native, seen = calls
    t = _tensors()
    w = {k: wrap(v) if v.is_floating_point() else v for k, v in t.items()}
    native.attn_append(0, w["q"], w["k"], w["v"], w["kp"], w["vp"], w["table"], [1, 2], [1, 2], w["out"], None, w["ws"], 0)
    args = seen[0][1]
    assert seen[0][0] == "agx_attn_prefixed_append"
    assert args[1:6] == tuple(t[k].data_ptr() for k in ("q", "k", "v", "kp", "vp"))
    assert args[6:9] == (5, t["table"].data_ptr(), 7) and args[11] == 2
    assert args[12:] == (t["out"].data_ptr(), None, t["ws"].data_ptr(), 400, None)
    logits = torch.zeros(3, 12)[:, :9]
    native.accept(0, wrap(logits), 1, 9, None, t["table"][0], None, None, None, None, w["ws"], 0)
    assert seen[1][1][1:5] == (logits.data_ptr(), 1, 12, 9) and seen[1][1][7:9] == (6, 3)


@pytest.mark.parametrize("form", [lambda n: n, float, np.int64, np.float32, lambda n: torch.tensor(n)], ids=["int", "float", "np_int", "np_float", "tensor"])
def test_sizes_are_whatever_int_takes(calls, form):
    native, seen = calls
    t = _tensors()
    logits = torch.zeros(3, 12)
    native.accept(0, logits, 1, form(9), None, t["table"][0], None, None, None, None, t["ws"], 0)
    assert seen[0][1][4] == 9


@pytest.mark.parametrize("shape", [(2,), (2, 1), (2, 3), (1,)])
def test_the_number_of_lengths_is_their_first_dimension(calls, shape):
    native, seen = calls
    t = _tensors()
    lengths = np.ones(shape, dtype=np.int32)
    native.attn(0, t["q"], None, None, t["kp"], t["vp"], t["table"], lengths, lengths.tolist(), t["out"], None, t["ws"], 0)
    assert seen[0][1][9] == shape[0]


def test_no_sequences_need_no_rows_and_one_append_without_rows_reaches_the_library(calls):
    native, seen = calls
    t = _tensors()
    for lengths in ([], [1]):
        native.attn_append(0, t["q"], None, None, t["kp"], t["vp"], t["table"], lengths, lengths, t["out"], None, None, 0)
    assert [(name, a[2], a[3], a[11]) for name, a in seen] == [("agx_attn_prefixed_append", None, None, 0), ("agx_attn_prefixed_append", None, None, 1)]


@pytest.mark.parametrize("bad", [b"bytes", bytearray(8), [1.0], 3, memoryview(b"x")])
def test_what_has_no_address_is_refused(calls, bad):
    native, seen = calls
    t = _tensors()
    with pytest.raises((TypeError, AttributeError)):
        native.attn(0, bad, None, None, t["kp"], t["vp"], t["table"], [1], [1], t["out"], None, t["ws"], 0)
    with pytest.raises(TypeError):
        native.attn(0, t["q"], None, None, np.zeros((5, 2)), t["vp"], t["table"], [1], [1], t["out"], None, t["ws"], 0)
    assert not seen


@pytest.mark.parametrize("array", [np.zeros((3, 4)), np.zeros((3, 4), order="F"), np.zeros(8)[::-2], np.zeros(0, np.float32), np.zeros(4, "V2")])
def test_addresses_of_host_arrays(calls, array):
    native, seen = calls
    t = _tensors()
    native.step(0, False, t["kp"], t["vp"], t["table"], [1], [1], array, t["k"], t["v"], None, 0, 9, 0, None, t["out"], None, None, None, t["ws"], 0)
    assert (seen[0][1][9] or 0) == array.ctypes.data


def test_the_module_belongs_to_one_version_of_torch(monkeypatch):
    """It uses torch's C++ classes: another torch makes it stale for the build, and unusable until it is built again."""
    from paper_2605_10380_b200 import build
    agx._binding()
    assert not build._binding_stale()
    monkeypatch.setattr(torch, "__version__", "1.2.3+cu99")
    assert build._binding_stale()
    monkeypatch.setattr(agx, "_native", None)
    with pytest.raises(RuntimeError, match="1.2.3"):
        agx._binding()
