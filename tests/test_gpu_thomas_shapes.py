"""The float32 modal Thomas kernel of the mixed path in its 256- and 128-thread
launch shapes, which it takes for about 4,900 lines and 9,800 (csrc/mixed.cu
thomas_shape): every segment length, with padding rows and without, by the bars of
the test of the 512-thread shape."""
import ctypes as C

import numpy as np
import pytest
import torch

import oracle as O
import seeded_inputs as S
from _tpt import load
from test_gpu_mixed import PRECS, _line_errors, _thomas_f32_sequential

pytestmark = pytest.mark.gpu
tpt, L = load()

# 5,600 lines: 256 threads, segments of 12, 16, 24 and 32 rows; 9,800: 128 threads
CASES = [((100, 50), nz) for nz in (30, 96, 127, 144, 191, 256)] + [((175, 50), nz) for nz in (5, 48, 61, 96, 113, 128)]


@pytest.mark.parametrize("lines,nz", CASES)
@pytest.mark.parametrize("prec", ["bf16x3", "tf32"])
@pytest.mark.parametrize("coef", [(1.0, -5e-4), (0.0, 1.0)])
def test_narrow_thomas_shapes_match_the_oracle_recurrence(lines, nz, prec, coef):
    n = lines + (nz,)
    bcs = [(1, 1)] * 3
    dirs = O.make_dirs(n, (1.5, 2.0, 2.5), bcs)
    plan = tpt.Plan(n, [d.dxf for d in dirs], [d.dxc for d in dirs], bcs, xform=(tpt.GEMM, tpt.GEMM),
                    alpha=coef[0], beta=coef[1], precision=PRECS[prec], rtol=1e-10, max_refine=30)
    plan.set_thomas_kernel(1)
    fh = S.uniform_rhs(n, 31).astype(np.float32).astype(np.float64)
    sing = O.is_singular(dirs, coef[0])
    nx, ny = lines
    ldy = (ny + 7) // 8 * 8
    t2 = np.zeros((nz, nx, ldy), np.float32)
    t2[:, :, :ny] = fh.transpose(2, 0, 1)
    t2d = torch.from_numpy(t2.ravel()).cuda()
    split = prec == "bf16x3"
    out = [torch.zeros(t2.size, dtype=torch.bfloat16 if split else torch.float32, device="cuda") for _ in range(2)]
    work = plan.new_workspace()
    st = L.lib.tpt_mixed_thomas(plan._h, C.c_void_p(t2d.data_ptr()), C.c_void_p(out[0].data_ptr()),
                                C.c_void_p(out[1].data_ptr() if split else 0), C.c_void_p(work.data_ptr()),
                                C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == L.TPT_OK, L.lib.tpt_status_string(st)
    got = (out[0].double() + out[1].double()).cpu().numpy().reshape(nz, nx, ldy)[:, :, :ny].transpose(1, 2, 0)
    w, ref_in = dirs[2].dxf, fh.copy()
    if sing:
        ref_in[0, 0, :] -= np.sum(w * ref_in[0, 0, :]) / np.sum(w)
    lx, ly = plan.eigenvalues(0), plan.eigenvalues(1)
    ref = O.thomas_modal(ref_in, lx, ly, dirs[2], coef[0], coef[1], (0, 0) if sing else None)
    seq = _thomas_f32_sequential(ref_in, lx, ly, dirs[2], coef[0], coef[1])
    if sing:
        ref[0, 0, :] -= np.sum(w * ref[0, 0, :]) / np.sum(w)
        seq[0, 0, :] = ref[0, 0, :]
    e_got, e_seq = _line_errors(got, ref), _line_errors(seq, ref)
    fmt = 2.0 ** -16 if split else 0.0
    assert np.all(e_got <= 16.0 * e_seq + 4e-6 + fmt), (e_got.max(), e_seq.max())
    assert np.median(e_got) <= 2.0 * np.median(e_seq) + 1e-6 + fmt / 2
    if sing:
        assert e_got[0, 0] <= 1e-7 + fmt, e_got[0, 0]
