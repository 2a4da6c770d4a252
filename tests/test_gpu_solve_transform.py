"""The transforms of a float64 plan's solves by themselves (csrc/residue.cu): long
contractions, whose moduli and paddings an Ozaki plan does not reach, and the
Fourier matrices of uniform directions, element by element against the matrices
applied in extended precision.  Tolerance as in test_gpu_residue, plus a quarter of
it for the rounding of the tabulated cosines and sines."""
import numpy as np
import pytest
import torch

import oracle as O
import seeded_inputs as S
from _tpt import load
from test_gpu_residue import _matrix, _plan, _rhs

pytestmark = pytest.mark.gpu
tpt, L = load()


def _check(A, plan, f, n, ax, inverse, room=1.0):
    out = plan.solve_transform(tpt.field_to_device(f), ax, inverse, plan.new_workspace())
    g = np.moveaxis(tpt.field_to_host(out, n), ax, 0).reshape(n[ax], -1)[:, :16]
    b = np.moveaxis(f, ax, 0).reshape(n[ax], -1)[:, :16]
    ref = A.astype(np.longdouble) @ b.astype(np.longdouble)
    aA, aB = np.abs(A).astype(np.float64), np.abs(b)
    tol = room * 2.0 ** -53 * (np.abs(ref) + np.outer(aA.sum(1), aB.max(0)) + np.outer(aA.max(1), aB.sum(0)))
    bad = np.abs(g - ref) > tol
    assert not bad.any(), (n, ax, inverse, int(bad.sum()), float((np.abs(g - ref) / tol).max()))


@pytest.mark.parametrize("n,ax", [((577, 12, 3), 0), ((1025, 9, 4), 0), ((2048, 6, 5), 0), ((11, 1000, 3), 1),
                                  ((12, 2048, 2), 1), ((274, 20, 4), 0), ((9, 279, 5), 1)])
def test_long_contractions(n, ax):
    _, plan = _plan(n, L.TPT_PREC_FP64)
    for inverse in (False, True):
        A = _matrix(plan, n, ax, inverse)
        for kind in ("noise", "decaying", "constant"):
            _check(A, plan, _rhs(n, kind), n, ax, inverse)


def _fourier(n, kind, inverse):
    """Rows of the real DFT in half-complex order (kind "periodic") or of the DCT-II, or of their inverses."""
    pi = np.longdouble("3.141592653589793238462643383279502884")
    k, i = np.arange(n, dtype=np.int64)[:, None], np.arange(n, dtype=np.int64)[None, :]
    if kind == "periodic":
        ang = 2 * pi * (((k + 1) // 2 * i) % n).astype(np.longdouble) / n
        A = np.where(k % 2 == 1, np.cos(ang), np.sin(ang))
        A[0] = 1.0
        A[n - 1] = np.where(np.arange(n) % 2, -1.0, 1.0)
        norm = np.full(n, np.longdouble(2) / n)
        norm[0] = norm[n - 1] = np.longdouble(1) / n
    else:
        A = np.cos(pi * ((k * (2 * i + 1)) % (4 * n)).astype(np.longdouble) / (2 * n))
        norm = np.full(n, np.longdouble(2) / n)
        norm[0] = np.longdouble(1) / n
    return (A * norm[:, None]).T if inverse else A


@pytest.mark.parametrize("m", [32, 256, 1024])
@pytest.mark.parametrize("kind", ["periodic", "neumann"])
@pytest.mark.parametrize("ax", [0, 1])
def test_fourier_matrices(m, kind, ax):
    n = (m, 10, 3) if ax == 0 else (10, m, 3)
    bc = (0, 0) if kind == "periodic" else (1, 1)
    bcs = [(1, 1)] * 3
    bcs[ax] = bc
    grids = [O.uniform_grid(n[a]) if a == ax else O.tanh_grid(n[a], 1.0, 1.5) for a in range(3)]
    plan = tpt.Plan(n, [g[0] for g in grids], [g[1] for g in grids], bcs, alpha=1.0, beta=-5e-4)
    assert plan.transforms()[ax] == tpt.FFT
    for inverse in (False, True):
        A = _fourier(m, kind, inverse)
        for f in (_rhs(n, "noise"), _rhs(n, "decaying")):
            _check(A, plan, f, n, ax, inverse, room=1.25)
        # and the plan's own Fourier transform computes the same matrix
        f = _rhs(n, "noise")
        fft = tpt.field_to_host(plan.transform(tpt.field_to_device(f), ax, inverse), n)
        fft, b = (np.moveaxis(v, ax, 0).reshape(m, -1)[:, :8] for v in (fft, f))
        ref = A @ b.astype(np.longdouble)
        assert np.abs(fft - ref).max() <= 1e-13 * np.abs(ref).max()
