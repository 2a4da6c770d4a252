"""The residue tables of a float64 plan's matrices belong to the cached direction,
like its other tables: plans that share a direction, in x or in y, share them, and
they count in the cache's bytes."""
import numpy as np
import pytest
import torch

import oracle as O
import seeded_inputs as S
from _tpt import load

pytestmark = pytest.mark.gpu
tpt, L = load()


@pytest.mark.parametrize("prec", [L.TPT_PREC_FP64, L.TPT_PREC_FP64_OZAKI])
@pytest.mark.parametrize("stretch,bc", [(1.5, (1, 1)), (0.0, (0, 0))])
def test_cached_plans_share_residue_tables(prec, stretch, bc):
    m = 128
    bcs = [bc, bc, (1, 1)]
    grid = O.uniform_grid(m) if stretch == 0.0 else O.tanh_grid(m, 1.0, stretch)
    d, dz = O.Direction(*grid, bc), O.Direction(*O.tanh_grid(20, 1.0, 1.5), (1, 1))
    n = (m, m, 20)
    spec = dict(n=n, dxf=[d.dxf, d.dxf, dz.dxf], dxc=[d.dxc, d.dxc, dz.dxc], bc=bcs, alpha=1.0, beta=-5e-4,
                precision=prec, max_refine=1)
    cache = tpt.Cache(0)
    f = tpt.field_to_device(S.uniform_rhs(n, 3))
    first = tpt.Plan(cache=cache, **spec)
    held = cache.stats()["device_bytes"]
    tables = 2 * m * 13 * 128 * 2               # forward and inverse, 13 moduli or more, K padded to 128
    assert held >= tables
    free = torch.cuda.mem_get_info()[0]
    more = [tpt.Plan(cache=cache, **dict(spec, beta=-1e-3 * i)) for i in range(1, 9)]
    assert cache.stats()["device_bytes"] == held
    assert free - torch.cuda.mem_get_info()[0] < 8 * tables
    own, _ = tpt.Plan(**spec).solve(f)
    assert torch.equal(first.solve(f)[0], own)
    ref, _ = O.solve_tensor(S.uniform_rhs(n, 3), [d, d, dz], 1.0, -1e-3)
    got = tpt.field_to_host(more[0].solve(f)[0], n)
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
    del first, more
