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
