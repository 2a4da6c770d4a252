"""Float64 solves through the residue transforms against the same plans on the
float64 FMA GEMM and the FFT (tpt_plan_limit_scratch 0), over the forms that both
accept: every boundary pair, uniform and stretched directions, directions outside
the operator, sizes on both sides of the residues' range and of their tiles, one
plane and many, out of place and in place, right-hand sides far from one.  Both
refine once against the same residual, so they differ by its rounding times the
condition number, below 1e-11 for these grids."""
import random

import pytest
import torch

import oracle as O
from _tpt import load

pytestmark = pytest.mark.gpu
tpt, L = load()

PAIRS = {"periodic": (0, 0), "neumann": (1, 1), "dirichlet": (2, 2), "mixed": (2, 1), "node": (3, 3), "none": (4, 4)}


def _form(seed):
    rng = random.Random(seed)
    n = [rng.choice((1, 2, 3, 16, 23, 24, 25, 31, 32, 33, 64, 65, 100, 127, 128, 130, 256, 257, 300)) for _ in range(2)]
    n.append(rng.choice((1, 2, 3, 9, 17, 33, 64, 100)))
    if n[0] * n[1] * n[2] > 2_000_000:
        n[2] = rng.choice((1, 3, 9, 17))
    bc = [rng.choice(("periodic", "neumann", "neumann", "dirichlet", "mixed", "node", "none")) for _ in range(2)]
    bc.append(rng.choice(("neumann", "neumann", "dirichlet", "mixed", "node")))
    stretch = [rng.choice((0.0, 0.0, 1.2, 2.5, 3.0)) for _ in range(3)]
    for a in range(3):
        if bc[a] == "periodic" and n[a] < 3:
            bc[a] = "neumann"
        if n[a] < 3 or (bc[a] == "periodic" and n[a] > 130):   # long cyclic eigenproblems are slow on the host
            stretch[a] = 0.0
    alpha, beta = rng.choice(((0.0, 1.0), (1.0, -5e-4), (1.0, -1e-2), (0.7, -1.3)))
    if "none" in bc and alpha == 0.0:
        alpha, beta = 1.0, -1e-3
    return n, [PAIRS[b] for b in bc], stretch, alpha, beta, rng.choice((1.0, 1.0, 1e200, 1e-200)), rng.random() < 0.3


@pytest.mark.parametrize("seed", range(60))
def test_residue_and_float64_transforms_agree(seed):
    n, bc, stretch, alpha, beta, scale, in_place = _form(seed)
    grids = [O.uniform_grid(m) if s == 0.0 else O.tanh_grid(m, 1.0, s) for m, s in zip(n, stretch)]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    for limit in (None, 0):
        plan = tpt.Plan(n, [g[0] for g in grids], [g[1] for g in grids], bc, alpha=alpha, beta=beta, max_refine=1)
        if limit is not None:
            plan.limit_scratch(limit)
        f = (torch.rand(plan.npts, dtype=torch.float64, device="cuda", generator=gen.manual_seed(seed)) - 0.5) * scale
        out.append(plan.solve(f, f)[0] if in_place else plan.solve(f)[0])
    worst = (out[0] - out[1]).abs().max().item()
    assert worst <= 1e-11 * out[1].abs().max().item(), _form(seed)
