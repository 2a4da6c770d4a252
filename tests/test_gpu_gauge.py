"""The canonical gauge of a singular float64 solve: the volume-weighted mean of phi
is removed to within 6 u of the mean of |phi| (csrc/kernels_fp64.cu), and the
subtraction rounds every value once more (u of it, and u of the mean taken off,
which is no larger than the mean of |phi| before it).  x-lines shorter and longer
than a warp's 32 and 64 values, odd lengths, few and many lines."""
import numpy as np
import pytest

import oracle as O
import seeded_inputs as S
from _tpt import load

pytestmark = pytest.mark.gpu
tpt, L = load()

U = 2.0 ** -53


@pytest.mark.parametrize("n", [(1, 1, 40), (2, 3, 5), (31, 9, 4), (33, 7, 6), (64, 5, 3), (97, 40, 33), (700, 5, 4),
                               (2051, 3, 2)])
def test_the_weighted_mean_is_removed_to_a_few_ulps(n):
    bcs = [(1, 1)] * 3
    dirs = O.make_dirs(n, (2.5, 1.5, 2.0), bcs)
    f = S.remove_weighted_mean(S.uniform_rhs(n, 2), [d.dxf for d in dirs])
    plan = tpt.Plan(n, [d.dxf for d in dirs], [d.dxc for d in dirs], bcs, max_refine=1)
    phi = tpt.field_to_host(plan.solve(tpt.field_to_device(f))[0], n).astype(np.longdouble)
    w = dirs[0].dxf.astype(np.longdouble)[:, None, None] * dirs[1].dxf[None, :, None] * dirs[2].dxf[None, None, :]
    mean, size = (w * phi).sum() / w.sum(), (w * np.abs(phi)).sum() / w.sum()
    assert abs(mean) <= 10 * U * size, (n, float(abs(mean) / (U * size)))
