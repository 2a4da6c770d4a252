"""The moduli of the residue transforms (csrc/residue.cu), for every contraction
length: pairwise coprime, and the tensor-core products exact.  The residues of the
data are r = v - p rint(v * float32(1 / p)), which can pass p / 2 near a tie of
large v; the values next to every tie within reach are tried here, in arithmetic
of this file's own."""
import ctypes as C
import functools
from math import gcd

import numpy as np
import pytest

from _tpt import load

tpt, L = load()

MATRIX_BITS, DATA_BITS, UP = 54, 53, 15     # csrc/residue.h


def _moduli(K):
    buf, cnt = (C.c_int * 18)(), C.c_int()
    assert L.lib.tpt_test_residue_moduli(K, buf, C.byref(cnt)) == L.TPT_OK
    return list(buf[:cnt.value])


def _centred(v, p):
    v %= p
    return v - p if 2 * v > p else v


@functools.lru_cache(None)
def _largest_residue(p):
    """max |r| over |v| <= the largest sum of digits (14 bits balanced, the top one 15 bits) times constants."""
    reach = max(sum((8192 if j < 3 else 32768) * abs(_centred(1 << (k + 14 * j), p)) for j in range(4))
                for k in range(UP + 1))
    tie = np.arange(0, reach // p + 1) * p + p // 2
    v = (tie[:, None] + np.arange(-2, 4)[None, :]).ravel()
    v = v[v <= reach].astype(np.float64)    # r is odd in v
    q = np.rint(v * float(np.float32(1.0) / np.float32(p)))   # 24 x 24 bits: exact in float64
    return int(np.abs(v - q * p).max())


@pytest.mark.parametrize("block", range(8))
def test_products_and_sums_are_exact(block):
    for K in range(1 + 256 * block, 257 + 256 * block):
        ps = _moduli(K)
        P = 1
        for i, p in enumerate(ps):
            assert all(gcd(p, q) == 1 for q in ps[:i])
            r = _largest_residue(p)
            assert r <= 256 and r * (p // 2) * K <= 1 << 24, (K, p, r)
            P *= p
        # |x| <= K 2^53 (2^54 P / 2^L + 1/2) < P / 2
        bits = P.bit_length()
        assert 2 * K * 2 ** DATA_BITS * (2 ** (MATRIX_BITS + 1) * P + 2 ** bits) < P * 2 ** (bits + 1), K


def test_lengths_out_of_range_are_refused():
    buf, cnt = (C.c_int * 18)(), C.c_int()
    for K in (0, -1, 2049):
        assert L.lib.tpt_test_residue_moduli(K, buf, C.byref(cnt)) == L.TPT_ERR_INVALID_ARG
