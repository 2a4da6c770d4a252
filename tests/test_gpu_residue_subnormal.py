"""Residue transforms of fields below the float64 normal range (csrc/residue.cu):
lines of subnormal values alone, and lines whose largest value is normal and
others not.  Tolerance as for the other fields, plus the spacing of subnormal
results."""
import numpy as np
import pytest

import seeded_inputs as S
from _tpt import load
from test_gpu_residue import _matrix, _plan

pytestmark = pytest.mark.gpu
tpt, L = load()


@pytest.mark.parametrize("n", [(15, 33, 4), (128, 70, 3), (257, 97, 2)])
@pytest.mark.parametrize("kind", ["subnormal", "straddling", "smallest"])
def test_transforms_below_the_normal_range(n, kind):
    _, p64 = _plan(n, L.TPT_PREC_FP64)
    _, poz = _plan(n, L.TPT_PREC_FP64_OZAKI)
    f = S.uniform_rhs(n, 7)
    if kind == "subnormal":
        f = np.ldexp(f, -1030)
    elif kind == "straddling":                       # 2^-1015 .. 2^-1045 along both axes
        i, j, _ = np.ogrid[:n[0], :n[1], :n[2]]
        f = np.ldexp(f, -1015 - (7 * i + 5 * j) % 31)
    else:                                            # zero or the smallest subnormal
        f = np.where(f > 0.5, 2.0 ** -1074, 0.0)
    assert (np.abs(f[f != 0]) < 2.0 ** -1022).any()
    for ax in (0, 1):
        for inverse in (False, True):
            A = _matrix(p64, n, ax, inverse)
            got = tpt.field_to_host(poz.transform(tpt.field_to_device(f), ax, inverse), n)
            g = np.moveaxis(got, ax, 0).reshape(n[ax], -1).astype(np.longdouble)
            b = np.moveaxis(f, ax, 0).reshape(n[ax], -1)
            aA, aB = np.abs(A).astype(np.longdouble), np.abs(b).astype(np.longdouble)
            ref = A.astype(np.longdouble) @ b.astype(np.longdouble)
            tol = np.longdouble(2) ** -53 * (np.abs(ref) + np.outer(aA.sum(1), aB.max(0)) +
                                             np.outer(aA.max(1), aB.sum(0))) + np.longdouble(2) ** -1074
            bad = np.abs(g - ref) > tol
            assert not bad.any(), (n, kind, ax, inverse, int(bad.sum()), float((np.abs(g - ref) / tol).max()))
