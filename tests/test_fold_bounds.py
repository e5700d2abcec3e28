"""Which primes the folded arithmetic accepts (hostmath::fold_consts), on the CPU: moduli at the very edge
of acceptance, for every width and both signs, keep each value a transform meets within the range that
one fold makes canonical.  The ranges are worked out here from what the kernels are handed."""
import ctypes
import re
import subprocess

import pytest


class FoldMod(ctypes.Structure):
    _fields_ = [("kc", ctypes.c_uint), ("mask", ctypes.c_uint), ("e", ctypes.c_int), ("big", ctypes.c_uint),
                ("kr", ctypes.c_uint), ("maskr", ctypes.c_uint), ("er", ctypes.c_int)]


@pytest.fixture(scope="module")
def consts():
    from paper_2312_04356_gb300 import build
    so = build.build()
    out = subprocess.run(["nm", "-D", "--defined-only", so], capture_output=True, text=True, check=True).stdout
    f = getattr(ctypes.CDLL(so), re.search(r"(\S*fold_consts\S*)", out).group(1))
    f.argtypes, f.restype = [ctypes.c_uint64, ctypes.POINTER(FoldMod)], ctypes.c_bool

    def call(q):
        m = FoldMod()
        return m if f(q, ctypes.byref(m)) else None
    return call


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("K", range(33, 61))
def test_values_at_the_edge_of_acceptance_stay_in_range(consts, K, sign):
    lo, hi = 0, 1 << 26                       # |e|: the largest accepted
    while hi - lo > 1:
        mid = (lo + hi) // 2
        m = consts((1 << K) - sign * mid)
        lo, hi = (mid, hi) if m and m.kc + 32 == K else (lo, mid)
    if lo == 0:
        assert K == 57                        # 128-bit sums of 57-bit primes do not fit
        return
    q, e = (1 << K) - sign * lo, lo
    big = consts(q).big
    R = (1 << K) + (e << 31)                  # a folded product
    # words a transform takes: residues, a conversion's, the centred lift of a residue below 2^61
    first = max(q, (1 << K) + (e << 16), (1 << K) + (e << 60 >> K))
    # a value opened by one fold, of any word a group of stages can end with
    limit = 7 << 60
    opened = (1 << K) + ((limit >> K) + 1) * e
    top = max(first, opened + 4 * R) if big else first + 16 * R
    assert top + q <= limit                   # a tail takes a residue minus it
    assert (4 if big else 16) * max(R, opened) <= limit        # sums of the inverse between folds
    assert ((top >> K) + 1) * e < q           # one fold leaves (-q, 2 q)
