"""Float64 Thomas (csrc/kernels_fp64.cu) at the ends of its launch rules: two
threads per line for few lines (shortest lines, odd and even, and the longest
whose z rows are staged in shared memory), one thread per line for many lines,
rows read from memory beyond 2048 points, first and later corrections.

A line's system is weakly diagonally dominant, so elimination from either end
satisfies (A + E) x = f with |E| <= 12 u |A| (4 u |L||U|, |L||U| <= 3 |A|); the
reciprocal pivots and the rounding of the beta-scaled rows and of the modal
shift add less than 20 u |A|.  Each row is held to 32 u (|A||x| + |f|)."""
import numpy as np
import pytest

import oracle as O
import seeded_inputs as S
from _tpt import load

import torch

pytestmark = pytest.mark.gpu
tpt, L = load()

U = 2.0 ** -53


def _plan(n, alpha, beta, **kw):
    dirs = O.make_dirs(n, (1.5, 2.0, 1.5), [(1, 1)] * 3)
    return dirs, tpt.Plan(n, [d.dxf for d in dirs], [d.dxc for d in dirs], [(1, 1)] * 3, xform=(tpt.GEMM, tpt.GEMM),
                          alpha=alpha, beta=beta, **kw)


def _rows(x, d, shift, beta):
    """(beta T_z + shift) x and the same with absolute values, in extended precision."""
    ld = np.longdouble
    a, b, c = (beta * v.astype(ld) for v in (d.a, d.b, d.c))
    x = x.astype(ld)
    lo, up = np.zeros_like(x), np.zeros_like(x)
    lo[..., 1:], up[..., :-1] = x[..., :-1], x[..., 1:]
    diag = b + shift[..., None].astype(ld)
    return a * lo + diag * x + c * up, abs(a * lo) + abs(diag * x) + abs(c * up)


# two threads a line, and 20,000 lines: one (which takes no static shared memory)
SIZES = [(5, 7, nz) for nz in (1, 2, 3, 8, 9, 33, 1962, 1963, 2048, 2049)] + [(160, 125, nz) for nz in (1, 2, 3, 8, 9, 33)]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("coef", [(0.0, 1.0), (1.0, -5e-4)])
def test_lines_satisfy_their_rows(n, coef):
    nz = n[2]
    dirs, plan = _plan(n, *coef)
    f = S.uniform_rhs(n, 21)
    x = tpt.field_to_host(plan.thomas(tpt.field_to_device(f)), n)
    lam = plan.eigenvalues(0)[:, None] + plan.eigenvalues(1)[None, :]
    null = (0, 0) if O.is_singular(dirs, coef[0]) else None
    if null is not None:            # the null line's right-hand side is projected, its solution centred
        w = dirs[2].dxf
        f[0, 0] -= np.sum(w * f[0, 0]) / np.sum(w)
        assert abs(np.sum(w * x[0, 0])) <= 4 * nz * U * np.sum(w * np.abs(x[0, 0]))
    Ax, absAx = _rows(x, dirs[2], coef[0] + coef[1] * lam, coef[1])
    err, tol = np.abs(Ax - f), 32 * U * (absAx + np.abs(f))
    if null is not None:            # its last row holds by compatibility: the sum of the others' rounding
        tol[0, 0] = 4 * nz * U * (absAx[0, 0] + np.abs(f[0, 0])).max()
    assert (err <= tol).all(), (n, coef, float((err / tol).max()))


@pytest.mark.parametrize("n", [(5, 7, 2), (30, 26, 3), (5, 7, 1963), (26, 30, 2048), (5, 7, 2049)])
def test_solves_with_kept_pivots_match_the_oracle(n):
    """Two corrections: the second reads the first one's pivots.  The coefficients
    keep the condition number below 100, so 1e-12 is 40 times eps cond."""
    dirs, plan = _plan(n, 1.0, -1e-6, max_refine=1)
    f = S.uniform_rhs(n, 6)
    phi, _ = plan.solve(tpt.field_to_device(f))
    torch.cuda.synchronize()
    ref, _ = O.solve_tensor(f, dirs, 1.0, -1e-6)
    assert np.abs(tpt.field_to_host(phi, n) - ref).max() <= 1e-12 * np.abs(ref).max()
