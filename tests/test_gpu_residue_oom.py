"""Float64 plan creation where the residue tables of the transform matrices find no
device memory: the plan takes the float64 FMA GEMM, which needs none, as such
plans did before they had tables."""
import ctypes as C

import numpy as np
import pytest

import oracle as O
import seeded_inputs as S
from _tpt import load

pytestmark = pytest.mark.gpu
tpt, L = load()

NNN = [(1, 1)] * 3


def test_plans_without_room_for_the_tables_take_the_float64_transforms():
    n = (40, 36, 28)
    dirs = O.make_dirs(n, (1.5, 2.0, 2.5), NNN)
    desc, keep = tpt.make_desc(n, [d.dxf for d in dirs], [d.dxc for d in dirs], NNN, alpha=1.0, beta=-5e-4)
    for after in range(100):
        h = C.c_void_p()
        try:
            L.lib.tpt_test_fail_allocations(after)
            st = L.lib.tpt_plan_create(C.byref(desc), 0, C.byref(h))
        finally:
            L.lib.tpt_test_fail_allocations(-1)
        if st == L.TPT_OK:
            break
        assert st == L.TPT_ERR_OOM and not h.value
    assert st == L.TPT_OK                        # every table but the residues
    plan = tpt.Plan.borrowed(h, n, 0)
    assert plan.workspace_bytes == 256 + 4 * 8 * int(np.prod(n))
    f = S.uniform_rhs(n, 5)
    got = tpt.field_to_host(plan.solve(tpt.field_to_device(f))[0], n)
    ref, _ = O.solve_tensor(f, dirs, 1.0, -5e-4)
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
    L.lib.tpt_plan_destroy(h)
