"""Rounding of the float64 residual kernel (csrc/kernels_fp64.cu), point by point:
every operation rounds once, so the error is at most u times the sum of the
partial sums' magnitudes in the kernel's order, x- d x+ | y- d y+ | z- d z+, then
f - alpha phi less beta times that.  On smooth fields those partial sums are small, and another order (f first,
or the six neighbours before the diagonals) exceeds the bound many times.  Sizes:
one block and several, several z segments, ragged edges, z rows from memory."""
import numpy as np
import pytest

import oracle as O
import seeded_inputs as S
from _tpt import load

pytestmark = pytest.mark.gpu
tpt, L = load()

U = 2.0 ** -53


def _partials(f, phi, dirs, alpha, beta):
    ld = np.longdouble
    f, phi = f.astype(ld), phi.astype(ld)
    terms = {}
    for ax, d in enumerate(dirs):
        shape = [1, 1, 1]
        shape[ax] = d.n
        a, b, c = (v.astype(ld).reshape(shape) for v in (d.a, d.b, d.c))
        terms[ax] = (a * np.roll(phi, 1, ax), b * phi, c * np.roll(phi, -1, ax))
    seq = [t for ax in range(3) for t in terms[ax]]
    acc, total = np.zeros_like(f), np.zeros_like(f)
    for t in seq:
        acc = acc + t
        total += np.abs(acc)
    rest = f - ld(alpha) * phi
    r = rest - ld(beta) * acc
    return r, abs(beta) * total + (np.abs(rest) if alpha else 0.0) + np.abs(r)


@pytest.mark.parametrize("n", [(64, 64, 64), (33, 6, 1), (1, 9, 50), (70, 45, 130), (9, 5, 2100)])
@pytest.mark.parametrize("kind", ["smooth", "noise"])
@pytest.mark.parametrize("stretch", [0.0, 2.0])
@pytest.mark.parametrize("alpha,beta", [(0.0, 1.0), (1.0, -5e-4)])
def test_residual_rounds_as_its_order_allows(n, kind, stretch, alpha, beta):
    dirs = O.make_dirs(n, (stretch,) * 3, [(2, 1), (1, 1), (2, 2)])
    if kind == "noise":
        phi = S.uniform_rhs(n, 3)
    else:
        x, y, z = ((np.arange(m) + 0.37) / m for m in n)
        phi = np.sin(1.3 * x)[:, None, None] + np.cos(2.1 * y)[None, :, None] * np.exp(-z)[None, None, :]
    f = S.uniform_rhs(n, 4)
    plan = tpt.Plan(n, [d.dxf for d in dirs], [d.dxc for d in dirs], [d.bc for d in dirs], xform=(tpt.GEMM,) * 2,
                    alpha=alpha, beta=beta)
    got = tpt.field_to_host(plan.residual(tpt.field_to_device(f), tpt.field_to_device(phi)), n)
    ref, total = _partials(f, phi, dirs, alpha, beta)
    ratio = (np.abs(got - ref) / (1.001 * U * total)).max()
    assert ratio <= 1.0, (n, kind, stretch, alpha, float(ratio))
