"""tpt_plan_limit_scratch: less workspace for a float64 plan or batch with the same
results, and float64 operands throughout at 0."""
import numpy as np
import pytest
import torch

import oracle as O
import seeded_inputs as S
from _tpt import load

pytestmark = pytest.mark.gpu
tpt, L = load()

NNN = [(1, 1)] * 3


def _spec(n, prec=L.TPT_PREC_FP64, stretch=(1.5, 2.0, 2.5), **kw):
    dirs = O.make_dirs(n, stretch, NNN)
    return dirs, dict(dict(n=n, dxf=[d.dxf for d in dirs], dxc=[d.dxc for d in dirs], bc=NNN, alpha=1.0, beta=-5e-4,
                           precision=prec, max_refine=1), **kw)


def _base(n):
    return 256 + 4 * ((8 * int(np.prod(n)) + 255) // 256 * 256)


@pytest.mark.parametrize("n,stretch", [((70, 45, 33), (1.5, 2.0, 2.5)), ((64, 48, 20), (0.0, 2.0, 2.5))])
def test_no_scratch_runs_the_float64_steps(n, stretch):
    """At 0 a solve without refinement is its single steps, bit by bit: the FMA GEMM
    of a stretched direction, the FFT of a uniform one."""
    _, spec = _spec(n, stretch=stretch, max_refine=0)
    plan = tpt.Plan(**spec)
    assert plan.workspace_bytes > _base(n)
    plan.limit_scratch(0)
    assert plan.workspace_bytes == _base(n)
    f = tpt.field_to_device(S.uniform_rhs(n, 5))
    t = plan.thomas(plan.transform(plan.transform(f, 0, False), 1, False))
    step = plan.transform(plan.transform(t, 1, True), 0, True)
    assert torch.equal(plan.solve(f, want_info=False)[0], step)


@pytest.mark.parametrize("prec", [L.TPT_PREC_FP64, L.TPT_PREC_FP64_OZAKI])
def test_smaller_passes_give_the_same_results(prec):
    n = (70, 45, 33)
    _, spec = _spec(n, prec)
    f = tpt.field_to_device(S.uniform_rhs(n, 5))
    plan = tpt.Plan(**spec)
    whole, size = plan.solve(f, want_info=False)[0], plan.workspace_bytes
    for limit in (size - _base(n) - 1, 1 << 20, 1 << 18):
        plan.limit_scratch(limit)
        assert _base(n) < plan.workspace_bytes <= _base(n) + limit
        assert torch.equal(plan.solve(f, want_info=False)[0], whole), limit
        small = plan.workspace_bytes
        plan.limit_scratch(1 << 40)
        assert plan.workspace_bytes == small
    plan.limit_scratch(0)
    if prec == L.TPT_PREC_FP64_OZAKI:            # one z plane stays
        assert _base(n) < plan.workspace_bytes <= small
        assert torch.equal(plan.solve(f, want_info=False)[0], whole)


def test_a_batch_shrinks_with_its_instances():
    sizes = [(70, 45, 33), (48, 64, 20), (33, 30, 50)]
    batch = tpt.Batch([_spec(n)[1] for n in sizes], nstreams=2)
    fs = [tpt.field_to_device(S.uniform_rhs(n, 5)) for n in sizes]
    refs = [O.solve_tensor(S.uniform_rhs(n, 5), _spec(n)[0], 1.0, -5e-4)[0] for n in sizes]
    before = batch.workspace_bytes
    work = batch.new_workspace()
    for limit in (None, 1 << 18, 0):
        if limit is not None:
            batch.limit_scratch(limit)
            assert batch.workspace_bytes < before
            work = batch.new_workspace()
        phis = [torch.zeros_like(f) for f in fs]
        for _ in range(2):                       # eager, then the recorded graph
            for p in phis:
                p.zero_()
            batch.solve(fs, phis, work)
            for p, n, r in zip(phis, sizes, refs):
                assert np.abs(tpt.field_to_host(p, n) - r).max() <= 1e-12 * np.abs(r).max()

