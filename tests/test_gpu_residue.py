"""Residue-number transform GEMMs (csrc/residue.cu) on GB300: one transform at a
time through an Ozaki plan's tpt_transform, against the float64 matrices applied
in extended precision, and float64 solves whose directions lie outside the Ozaki
plan's range, against the oracle.

Tolerance of an element x = sum_k a_k b_k, from the arithmetic: each operand row
is rounded to 2^-54 of its power-of-two scale (at most twice its maximum), the
fraction is kept to 2^-61 of at most 8 max|a| sum|b|, and the result is rounded
once: 2^-53 |x| + 2^-53 (max|b| sum|a| + max|a| sum|b|) covers their sum."""
import numpy as np
import pytest
import torch

import oracle as O
import seeded_inputs as S
from _tpt import load

pytestmark = pytest.mark.gpu
tpt, L = load()

NNN = [(1, 1)] * 3


def _plan(n, prec, bcs=NNN, alpha=0.0, beta=1.0, stretch=(1.5, 2.0, 2.5), **kw):
    dirs = O.make_dirs(n, stretch, bcs)
    return dirs, tpt.Plan(n, [d.dxf for d in dirs], [d.dxc for d in dirs], bcs, xform=(tpt.GEMM, tpt.GEMM),
                          alpha=alpha, beta=beta, precision=prec, **kw)


def _matrix(p64, n, ax, inverse):
    """The float64 transform matrix of direction ax: the transform of the unit vectors."""
    K = n[ax]
    e = np.zeros(n)
    cols = np.zeros((K, K))
    lines = [d for d in range(3) if d != ax]
    per = n[lines[0]] * n[lines[1]]
    for k0 in range(0, K, per):
        e[:] = 0.0
        m = np.moveaxis(e, ax, 0).reshape(K, -1)
        for k in range(k0, min(K, k0 + per)):
            m[k, k - k0] = 1.0
        e = np.moveaxis(m.reshape([K] + [n[d] for d in lines]), 0, ax)
        out = tpt.field_to_host(p64.transform(tpt.field_to_device(e), ax, inverse), n)
        o = np.moveaxis(out, ax, 0).reshape(K, -1)
        for k in range(k0, min(K, k0 + per)):
            cols[:, k] = o[:, k - k0]
    return cols


def _rhs(n, kind):
    f = S.uniform_rhs(n, 7)
    if kind == "decaying":     # a few large values, the rest far below them
        i, j, k = np.ogrid[:n[0], :n[1], :n[2]]
        f = f / ((1.0 + i) ** 2 * (1.0 + j) ** 2)
    elif kind == "scaled":     # every line on another power of ten, some beyond the float32 range
        i, j, k = np.ogrid[:n[0], :n[1], :n[2]]
        f = f * 10.0 ** (((i * 7 + j * 5 + k * 3) % 41) - 20.0) * 10.0 ** ((k % 3) * 60.0 - 60.0)
    elif kind == "constant":   # one sign, one value: the largest sums of residues
        f = np.full(n, -0.999999999)
    return f


# tiles are 128 x 128, K chunks 64, MMA steps 16; the moduli change above K = 256
SIZES = [(1, 5, 3), (15, 33, 9), (64, 65, 4), (127, 129, 2), (128, 256, 3), (257, 97, 5), (33, 512, 2), (512, 40, 7),
         (576, 31, 5)]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("kind", ["noise", "decaying", "scaled", "constant"])
def test_transforms_are_as_accurate_as_their_rounding(n, kind):
    _, p64 = _plan(n, L.TPT_PREC_FP64)
    _, poz = _plan(n, L.TPT_PREC_FP64_OZAKI)
    f = _rhs(n, kind)
    for ax in (0, 1):
        for inverse in (False, True):
            A = _matrix(p64, n, ax, inverse)
            got = tpt.field_to_host(poz.transform(tpt.field_to_device(f), ax, inverse), n)
            g = np.moveaxis(got, ax, 0).reshape(n[ax], -1)[:, :200]
            b = np.moveaxis(f, ax, 0).reshape(n[ax], -1)[:, :200]
            ref = A.astype(np.longdouble) @ b.astype(np.longdouble)
            aA, aB = np.abs(A), np.abs(b)
            tol = 2.0 ** -53 * (np.abs(ref) + np.outer(aA.sum(1), aB.max(0)) + np.outer(aA.max(1), aB.sum(0)))
            bad = np.abs(g - ref) > tol
            assert not bad.any(), (n, kind, ax, inverse, int(bad.sum()), float((np.abs(g - ref) / tol).max()))


def test_a_non_finite_line_gives_nan_and_leaves_the_others():
    n = (70, 45, 6)
    _, poz = _plan(n, L.TPT_PREC_FP64_OZAKI)
    f = S.uniform_rhs(n, 3)
    clean = f.copy()
    f[3, 4, 1], f[60, 44, 5] = np.inf, np.nan
    for ax in (0, 1):
        got = tpt.field_to_host(poz.transform(tpt.field_to_device(f), ax, False), n)
        ref = tpt.field_to_host(poz.transform(tpt.field_to_device(clean), ax, False), n)
        hit = np.zeros(n, bool)
        for i, j, k in ((3, 4, 1), (60, 44, 5)):
            hit[(slice(None), j, k) if ax == 0 else (i, slice(None), k)] = True
        assert np.isnan(got[hit]).all() and np.array_equal(got[~hit], ref[~hit])


def test_passes_over_planes_equal_single_planes():
    """A field whose residues exceed the scratch (512 MB: 29,000 z planes here)
    goes in passes of whole planes; its planes equal those of a small field."""
    n, m = (11, 11, 40000), (11, 11, 40)
    small, big = _plan(m, L.TPT_PREC_FP64_OZAKI)[1], _plan(n, L.TPT_PREC_FP64_OZAKI)[1]
    f = S.uniform_rhs(n, 9)
    for ax in (0, 1):
        got = tpt.field_to_host(big.transform(tpt.field_to_device(f), ax, False), n)
        for k0 in (0, 29280, 39960):
            ref = tpt.field_to_host(small.transform(tpt.field_to_device(f[:, :, k0:k0 + 40]), ax, False), m)
            assert np.array_equal(got[:, :, k0:k0 + 40], ref), (ax, k0)


@pytest.mark.parametrize("n", [(600, 20, 12), (12, 1030, 9), (2049, 6, 5)])
def test_float64_solves_of_long_directions_match_the_oracle(n):
    dirs, plan = _plan(n, L.TPT_PREC_FP64, alpha=1.0, beta=-5e-4, max_refine=1)
    f = S.uniform_rhs(n, 5)
    phi, info = plan.solve(tpt.field_to_device(f))
    ref, _ = O.solve_tensor(f, dirs, 1.0, -5e-4)
    assert np.abs(tpt.field_to_host(phi, n) - ref).max() <= 1e-12 * np.abs(ref).max()


def test_non_finite_right_hand_side_is_reported():
    n = (40, 36, 28)
    _, plan = _plan(n, L.TPT_PREC_FP64, alpha=1.0, beta=-5e-4, rtol=1e-10, max_refine=3)
    f = S.uniform_rhs(n, 5)
    f[1, 2, 3] = np.nan
    with pytest.raises(L.TptError) as e:
        plan.solve(tpt.field_to_device(f))
    assert e.value.status == L.TPT_ERR_NONFINITE


@pytest.mark.parametrize("spare", [0, 1 << 20])
def test_a_tight_server_budget_still_takes_a_float64_request(spare):
    """Fields and the four workspace regions alone (no room for residues), and
    room for a few planes of them: the request runs and equals its own solve."""
    n = (64, 48, 40)
    dirs, plan = _plan(n, L.TPT_PREC_FP64, alpha=1.0, beta=-5e-4, max_refine=1)
    f = S.uniform_rhs(n, 5)
    ref, _ = plan.solve(tpt.field_to_device(f))
    budget = 6 * 8 * int(np.prod(n)) + 8 * 256 + spare
    srv = tpt.Server(device=0, slots=1, setup_threads=1, memory_budget=budget)
    try:
        fh = tpt.field_to_device(f, "cpu").pin_memory()
        ph = torch.empty_like(fh).pin_memory()
        t = srv.submit(fh, ph, n=n, dxf=[d.dxf for d in dirs], dxc=[d.dxc for d in dirs], bc=NNN,
                       xform=(tpt.GEMM, tpt.GEMM), alpha=1.0, beta=-5e-4, precision=L.TPT_PREC_FP64, max_refine=1)
        res = srv.wait(t, timeout=60.0)
        assert res is not None and res["status"] == L.TPT_OK and res["device_bytes"] <= budget
        assert (ph - ref.cpu()).abs().max().item() <= 1e-12 * ref.abs().max().item()
    finally:
        srv.close()


# a uniform direction in a float64 solve takes its transform's matrix from 32 to
# 1024 points, the FFT outside that range: both ends, periodic and Neumann, in
# x and in y, against the oracle at the float64 bar
@pytest.mark.parametrize("n,bcs", [((32, 24, 20), [(0, 0), (1, 1), (1, 1)]), ((1024, 16, 6), [(1, 1)] * 3),
                                   ((24, 64, 20), [(1, 1), (0, 0), (2, 1)]), ((128, 128, 10), [(0, 0), (1, 1), (1, 1)]),
                                   ((16, 2048, 3), [(1, 1), (1, 1), (2, 2)])])
def test_uniform_directions_match_the_oracle(n, bcs):
    dirs = [O.Direction(*O.uniform_grid(n[a]), bcs[a]) if a < 2 else O.Direction(*O.tanh_grid(n[a], 1.0, 1.5), bcs[a])
            for a in range(3)]
    f = S.uniform_rhs(n, 4)
    if O.is_singular(dirs, 0.0):
        f = S.remove_weighted_mean(f, [d.dxf for d in dirs])
    plan = tpt.Plan(n, [d.dxf for d in dirs], [d.dxc for d in dirs], bcs, precision=L.TPT_PREC_FP64, max_refine=1)
    phi, _ = plan.solve(tpt.field_to_device(f))
    ref, _ = O.solve_tensor(f, dirs, 0.0, 1.0)
    assert np.abs(tpt.field_to_host(phi, n) - ref).max() <= 1e-12 * np.abs(ref).max()
