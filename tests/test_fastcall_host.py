"""The binding's marshalling extension, on the host: its signatures are those of
the ctypes prototypes, host offsets of any kind reach the C functions as int32,
and errors come back as before."""
import ctypes
import os
import re

import numpy as np
import pytest

from paper_2506_07416_gb300 import select

SRC = os.path.join(os.path.dirname(select.__file__), "csrc", "fastcall.c")
KIND = {ctypes.c_void_p: "hpn", ctypes.c_int32: "i", ctypes.c_int64: "l", ctypes.c_float: "f"}


def test_signatures_match_the_prototypes():
    text = open(SRC).read()
    names = re.findall(r'"(\w+)"', re.search(r"kNames\[F_COUNT\] = \{(.*?)\};", text, re.S).group(1))
    sigs = re.findall(r'"(\w*)"', re.search(r"kSigs\[F_COUNT\] = \{(.*?)\};", text, re.S).group(1))
    assert len(names) == len(sigs)
    for name, sig in zip(names, sigs):
        if sig:
            proto = getattr(select.LIB, "litevlm_select_" + name).argtypes
            assert len(proto) == len(sig), name
            for t, c in zip(proto, sig):
                assert c in KIND[t], (name, t, c)


@pytest.mark.parametrize("kind", [np.int32, np.int64, list, "strided", "tensor"])
def test_keep_total_of_any_offsets(kind):
    so = np.array([0, 100, 100, 357, 2000], np.int32)
    kk = np.array([3, 0, 257, 11], np.int32)

    def as_kind(a):
        if kind is list:
            return a.tolist()
        if kind == "strided":
            return np.repeat(a, 2)[::2]
        if kind == "tensor":
            return pytest.importorskip("torch").from_numpy(a.copy())
        return a.astype(kind)

    assert select._keep_total(as_kind(so), None, 0.3) == int(select.keep_offsets(so, None, 0.3)[-1])
    assert select._keep_total(as_kind(so), as_kind(kk), 0.0) == int(kk.sum())
    long = np.arange(0, 700, 7, dtype=np.int32)  # more requests than the extension's own buffer holds
    assert select._keep_total(long, None, 0.5) == int(select.keep_offsets(long, None, 0.5)[-1])


@pytest.fixture
def topk_args():
    """_FC.topk with a recorder in the place of the C function: the arguments it was called with."""
    seen = []
    proto = ctypes.CFUNCTYPE(ctypes.c_int, *select.LIB.litevlm_select_topk.argtypes)
    rec = proto(lambda *a: seen.append(a) or 0)
    names = ("score", "score_full_keys", "score_topk", "topk", "compact", "splice", "project", "keep_offsets")

    def bind(**over):
        addr = {n: ctypes.cast(getattr(select.LIB, "litevlm_select_" + n), ctypes.c_void_p).value for n in names}
        select._FC.bind({**addr, **over}, select._host_i32, np.ndarray, select._ctypes_value)

    bind(topk=ctypes.cast(rec, ctypes.c_void_p).value)
    yield lambda **kw: _topk(seen, **kw)
    bind()


def _topk(seen, handle=16, batch=2, scores=32, ratio=0.25, stream=48):
    seen.clear()
    assert select._FC.topk(handle, batch, scores, None, [0, 1, 2], None, None, ratio, 64, 80, None, stream) == 0
    a = seen[0]
    return dict(handle=a[0], batch=a[1], scores=a[2], ratio=a[7], stream=a[11])


def test_pointers_and_numbers(topk_args):
    """Device pointers: None, ints, arrays, objects with data_ptr(); handles and numbers as ctypes takes them."""
    torch = pytest.importorskip("torch")
    a, t = np.arange(5, dtype=np.float32), torch.arange(5)
    assert topk_args(scores=None)["scores"] is None
    assert topk_args(scores=a)["scores"] == a.ctypes.data
    assert topk_args(scores=a[1:])["scores"] == a.ctypes.data + 4
    assert topk_args(scores=a.view("datetime64[s]" if a.itemsize == 8 else "V4"))["scores"] == a.ctypes.data
    d = np.zeros(3, "datetime64[s]")  # a type without a buffer format
    assert topk_args(scores=d)["scores"] == d.ctypes.data
    assert topk_args(scores=t)["scores"] == t.data_ptr()
    assert topk_args(handle=ctypes.c_void_p(1 << 40))["handle"] == 1 << 40
    assert topk_args(handle=None, stream=ctypes.c_void_p(None)) == dict(topk_args(), handle=None, stream=None)
    for three in (3, np.int64(3), np.int32(3), np.array(3), torch.tensor(3), ctypes.c_int32(3), (1 << 70) + 3):
        assert topk_args(batch=three)["batch"] == 3
    for half in (0.5, np.float32(0.5), np.float64(0.5), torch.tensor(0.5), ctypes.c_float(0.5)):
        assert topk_args(ratio=half)["ratio"] == 0.5
    assert topk_args(ratio=-1.0)["ratio"] == -1.0


@pytest.mark.parametrize("o", [np.int64(16), np.uint64(16), np.float32(1), ctypes.c_void_p(16), ctypes.c_int64(16),
                               (ctypes.c_char * 64)(), b"abc", bytearray(64), memoryview(bytearray(64)), "abc", 1.0,
                               [16], object()], ids=lambda o: type(o).__name__)
def test_no_address_of_an_object_is_taken_for_a_pointer(topk_args, o):
    with pytest.raises(AttributeError):
        topk_args(scores=o)
    for n in range(3):  # kept_idx, a source, a destination of compact
        a = [16, [16], [16]]
        a[n] = o if n == 0 else [o]
        with pytest.raises(AttributeError):
            select.compact(None, 1, a[0], 1, a[1], a[2], [16], stream=0)
    if not isinstance(o, ctypes.c_void_p):
        with pytest.raises(TypeError):
            topk_args(handle=o)


@pytest.mark.parametrize("o", ["3", 1.5, None, ctypes.c_int64(3), ctypes.c_float(3)], ids=lambda o: type(o).__name__)
def test_no_whole_number(topk_args, o):
    with pytest.raises(TypeError):
        topk_args(batch=o)


def test_errors():
    with pytest.raises(select.LitevlmError) as e:
        select._keep_total(np.array([0, 5], np.int32), None, 1.5)
    assert e.value.name == "INVALID_ARG" and "keep_ratio" in str(e.value)
    with pytest.raises(select.LitevlmError) as e:  # a NULL handle, stream 0
        select.score(None, 1, 0, 0, [0, 1], 0, 0, [0, 1], 1.0, 1.0, 0, stream=0)
    assert e.value.name == "INVALID_ARG"
    with pytest.raises(TypeError):
        select._FC.score(None, 1)
    with pytest.raises(AttributeError):  # no pointer in it
        select.score(None, 1, object(), 0, [0, 1], 0, 0, [0, 1], 1.0, 1.0, 0, stream=0)
    for n in (0, 9):
        with pytest.raises(select.LitevlmError):
            select.compact(None, 1, 16, 1, [16] * n, [16] * n, [16] * n, stream=0)
