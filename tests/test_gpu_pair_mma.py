"""Transform GEMM tiles run by a pair of CTAs per MMA (csrc/gemm_tc.cu, split
bf16 operands, 256-column tiles, K >= 384, grids of at least two tiles per SM): ragged
edges and contractions of whole and partial K chunks, by exact integer products;
and a solve whose y transforms take them, against the oracle's residual and the
same plan on 128-column tiles."""
import ctypes as C

import numpy as np
import pytest
import torch

import oracle as O
import seeded_inputs as S
from _tpt import load

pytestmark = pytest.mark.gpu
tpt, L = load()


@pytest.mark.parametrize("kind", ["f32", "split"])
@pytest.mark.parametrize("tma_out", [0, 1])
@pytest.mark.parametrize("shape", [(40 * 128 - 5, 2048, 384), (40 * 128, 2500, 400), (200, 256 * 160, 520),
                                   (256, 256 * 152 + 8, 1000)])
def test_pair_mma_products_are_exact(shape, tma_out, kind):
    M, N, K = shape
    rng = np.random.default_rng(M + N + K)
    A = torch.from_numpy(rng.integers(-40, 41, size=(M, K)).astype(np.float64)).cuda()
    B = torch.from_numpy(rng.integers(-40, 41, size=(N, K)).astype(np.float64)).cuda()
    ld = (M + 7) // 8 * 8
    dt = torch.float32 if kind == "f32" else torch.bfloat16
    out = [torch.full((N * ld + 64,), -7.25, dtype=dt, device="cuda") for _ in range(2)]
    work = torch.empty(8 * (M + N) * (K + 8) + 1024, dtype=torch.uint8, device="cuda")
    st = L.lib.tpt_tc_gemm_out(L.TPT_PREC_MIXED_BF16X3, M, N, K, C.c_void_p(A.data_ptr()), C.c_void_p(B.data_ptr()),
                               L.TPT_GEMM_OUT_F32 if kind == "f32" else L.TPT_GEMM_OUT_SPLIT_BF16, 1 << 30, 0, ld,
                               C.c_void_p(out[0].data_ptr()), C.c_void_p(out[1].data_ptr()),
                               C.c_void_p(work.data_ptr()), C.c_void_p(torch.cuda.current_stream().cuda_stream),
                               256, tma_out, 0)
    assert st == L.TPT_OK
    torch.cuda.synchronize()
    ref = (B @ A.T)                                  # exact: |sum| < 2^24; element (n, m)
    got = [o[:N * ld].view(N, ld) for o in out]
    if kind == "f32":
        assert torch.equal(got[0][:, :M].double(), ref)
    else:
        hi = ref.to(torch.bfloat16)
        assert torch.equal(got[0][:, :M], hi)
        assert torch.equal(got[1][:, :M], (ref - hi.double()).to(torch.bfloat16))
    assert (out[0][N * ld:] == -7.25).all()


def test_a_solve_on_pair_mma_tiles():
    n = (256, 512, 160)
    bcs = [(1, 1)] * 3
    dirs = O.make_dirs(n, (1.5, 2.0, 2.5), bcs)
    f = S.remove_weighted_mean(S.uniform_rhs(n, 8), [d.dxf for d in dirs])
    plan = tpt.Plan(n, [d.dxf for d in dirs], [d.dxc for d in dirs], bcs, xform=(tpt.GEMM, tpt.GEMM),
                    precision=L.TPT_PREC_MIXED_BF16X3, rtol=1e-10, max_refine=30)
    fd = tpt.field_to_device(f)
    phi = tpt.field_to_host(plan.solve(fd)[0], n)
    r = O.residual(f, phi, dirs, 0.0, 1.0)
    assert np.linalg.norm(r) <= 2e-10 * np.linalg.norm(f)
    plan.set_tiles((128,) * 4)
    ref = tpt.field_to_host(plan.solve(fd)[0], n)
    assert np.abs(phi - ref).max() <= 1e-9 * np.abs(ref).max()
