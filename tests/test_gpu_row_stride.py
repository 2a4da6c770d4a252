"""Mixed solves of even Nx that is not a multiple of four: the float-pair planes
have padded rows so that the TMA-staged residual runs; against the oracle, the
direct-load residual and outputs that are not 16-byte aligned."""
import numpy as np
import pytest
import torch

import oracle as O
import seeded_inputs as S
from _tpt import load

pytestmark = pytest.mark.gpu
tpt, L = load()

CASES = [((2, 9, 5), [(1, 1)] * 3, (0.0, 1.0)), ((66, 20, 17), [(0, 0), (1, 1), (1, 1)], (0.0, 1.0)),
         ((126, 24, 33), [(2, 1), (0, 0), (2, 2)], (1.0, -5e-4)), ((130, 17, 70), [(1, 1)] * 3, (1.0, -5e-4))]


@pytest.mark.parametrize("prec", [L.TPT_PREC_MIXED_BF16X3, L.TPT_PREC_MIXED_TF32])
@pytest.mark.parametrize("case", CASES)
def test_padded_rows(case, prec):
    n, bcs, coef = case
    dirs = O.make_dirs(n, (1.5, 2.0, 2.5), bcs)
    f = S.uniform_rhs(n, 12)
    if O.is_singular(dirs, coef[0]):
        f = S.remove_weighted_mean(f, [d.dxf for d in dirs])
    ref, _ = O.solve_tensor(f, dirs, *coef)
    bar = 1e-9 * np.abs(ref).max()
    for variant in (0, 1):
        plan = tpt.Plan(n, [d.dxf for d in dirs], [d.dxc for d in dirs], bcs, xform=(tpt.GEMM, tpt.GEMM), alpha=coef[0],
                        beta=coef[1], precision=prec, rtol=1e-10, max_refine=40)
        plan.set_residual_kernel(variant)
        work = plan.new_workspace()
        work.fill_(255)                       # NaN in every padding column
        fd = tpt.field_to_device(f)
        got = tpt.field_to_host(plan.solve(fd, work=work)[0], n)
        assert np.abs(got - ref).max() <= bar
        odd_f = torch.empty(plan.npts + 1, dtype=torch.float64, device="cuda")[1:]   # 8-byte alignment
        odd_phi = torch.empty(plan.npts + 1, dtype=torch.float64, device="cuda")[1:]
        odd_f.copy_(fd)
        got = tpt.field_to_host(plan.solve(odd_f, odd_phi, work)[0], n)
        assert np.abs(got - ref).max() <= bar
