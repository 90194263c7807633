"""A batch's descriptors, packed directly, hold the bytes of GemmDesc objects built field by field,
for every kind of argument the general way takes; what it refuses is still refused."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2503_22875_gb300 import ozg

T = torch.zeros(16, dtype=torch.float64)
N = np.zeros(16)
BASE = ("N", "T", 3, 4, 5, 1.5, T, 6, T[3:], 7, -0.0, T[5:], 8)


def general(calls, address):
    arr = (ozg.GemmDesc * len(calls))()
    for i, (ta, tb, m, n, k, al, A, lda, B, ldb, be, C, ldc) in enumerate(calls):
        arr[i] = ozg.GemmDesc(ta.encode(), tb.encode(), b"", m, n, k, float(al), float(be), address(A), lda,
                              address(B), ldb, address(C), ldc)
    return arr


def put(**kw):
    names = ("ta", "tb", "m", "n", "k", "al", "A", "lda", "B", "ldb", "be", "C", "ldc")
    return tuple(kw.get(x, v) for x, v in zip(names, BASE))


VARIANTS = [put(), put(ta="t", tb="c"), put(ta="x"), put(m=-1), put(k=np.int64(4)), put(m=True), put(k=2 ** 63 - 1), put(k=2 ** 70), put(ldc=-2 ** 63),
            put(al=np.float64(0.1)), put(al=np.float32(0.1)), put(be=2), put(al=float("nan")), put(A=None), put(A=0),
            put(B=T.data_ptr() + 8), put(C=2 ** 64 - 1), put(C=-1), put(al="0.25")]
REFUSED = [put(m=1.0), put(ta="NN"), put(ta=1), put(al="a"), put(al=1j), put(m=None)]


@pytest.mark.parametrize("host", [False, True])
def test_packed_descriptors(host):
    quick, address = (ozg._hp, ozg._hp) if host else (ozg._data_ptr, ozg._p)
    calls = VARIANTS + ([put(A=N, C=N[2:])] if host else [])
    assert ozg._DESC.size == ctypes.sizeof(ozg.GemmDesc)
    assert bytes(ozg._descs(calls, quick, address)) == bytes(general(calls, address))
    for c in REFUSED + ([] if host else [put(A=N)]):
        with pytest.raises(Exception) as want:
            general([c], address)
        with pytest.raises(want.type):
            ozg._descs([put(), c], quick, address)
