"""A bounded wait that runs out in the tensor-core transforms of a float64 solve
(producers that issue no loads; no GPU fault involved) never passes for a result:
every form of the call reports it or leaves NaN, and the next solve is right."""
import ctypes as C

import numpy as np
import pytest
import torch

import oracle as O
import seeded_inputs as S
from _tpt import load

pytestmark = pytest.mark.gpu
tpt, L = load()

NNN = [(1, 1)] * 3
# one wave of tiles, and several tiles per CTA; singular and not
CASES = [((40, 36, 28), 0.0, 1.0), ((256, 200, 150), 1.0, -5e-4)]


def _spec(n, alpha, beta, rtol=0.0):
    dirs = O.make_dirs(n, (1.5, 2.0, 2.5), NNN)
    f = S.uniform_rhs(n, 5)
    f = S.remove_weighted_mean(f, [d.dxf for d in dirs]) if alpha == 0.0 else f
    return dirs, f, dict(n=n, dxf=[d.dxf for d in dirs], dxc=[d.dxc for d in dirs], bc=NNN, alpha=alpha, beta=beta,
                         precision=L.TPT_PREC_FP64, max_refine=1, rtol=rtol)


def _hook(plan, on):
    assert L.lib.tpt_test_transform_timeout(plan._h, on) == L.TPT_OK


@pytest.mark.parametrize("n,alpha,beta", CASES)
def test_a_timed_out_solve_is_not_taken_for_a_result(n, alpha, beta):
    dirs, f, spec = _spec(n, alpha, beta)
    plan = tpt.Plan(**spec)
    fd, phi = tpt.field_to_device(f), plan.new_field().fill_(7.0)
    good, _ = plan.solve(fd)
    _hook(plan, 1)
    plan.solve(fd, phi, want_info=False)
    assert torch.isnan(phi).all()                       # nobody reads a status here
    _, info = plan.solve(fd)
    assert np.isnan(info["rel_residual"])
    fh = tpt.field_to_device(f, "cpu").pin_memory()
    ph = torch.empty_like(fh).pin_memory()
    with pytest.raises(L.TptError) as e:
        plan.solve_host(fh, ph, plan.new_field(), plan.new_field(), plan.new_workspace())
    assert e.value.status == L.TPT_ERR_TIMEOUT
    _hook(plan, 0)
    again, _ = plan.solve(fd)
    # the residual's sums are atomics, the solution's arithmetic is not
    assert torch.equal(again, good)
    adaptive = tpt.Plan(**dict(spec, rtol=1e-10))
    _hook(adaptive, 1)
    with pytest.raises(L.TptError) as e:
        adaptive.solve(fd)
    assert e.value.status == L.TPT_ERR_TIMEOUT


def test_a_timed_out_instance_of_a_batch_is_reported():
    specs = [_spec((40, 36, 28), 0.0, 1.0), _spec((48, 32, 24), 1.0, -5e-4)]
    batch = tpt.Batch([s[2] for s in specs])
    fs = [tpt.field_to_device(s[1]) for s in specs]
    phis = [torch.zeros_like(f) for f in fs]
    work = batch.new_workspace()
    for on, want in ((0, L.TPT_OK), (1, L.TPT_ERR_TIMEOUT), (0, L.TPT_OK)):
        _hook(batch.plans[1], on)
        batch.solve(fs, phis, work, want_info=False)
        torch.cuda.synchronize()
        infos, st = (L.tpt_info * 2)(), (C.c_int * 2)()
        L.lib.tpt_batch_infos(batch._h, infos, st)
        assert list(st) == [L.TPT_OK, want]
        assert bool(torch.isnan(phis[1]).all()) == (want != L.TPT_OK)
        assert not torch.isnan(phis[0]).any()


def test_the_hook_refuses_plans_without_tensor_core_transforms():
    _, _, spec = _spec((8, 9, 10), 1.0, -5e-4)          # below 24 points: float64 FMA GEMM
    assert L.lib.tpt_test_transform_timeout(tpt.Plan(**spec)._h, 1) == L.TPT_ERR_INVALID_ARG
