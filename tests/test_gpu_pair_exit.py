"""Early exit of the transform GEMM whose MMAs run over pairs of CTAs: one CTA of
each pair stops loading after three stages (no GPU fault involved), so the two
have issued different numbers of stages.  The pair waits for the copies that were
issued before either CTA leaves, the call reports the timeout, and the kernels
that run next on the same shared memory give exact products."""
import ctypes as C

import pytest
import torch

from _tpt import load

pytestmark = pytest.mark.gpu
tpt, L = load()


def _exact_product(seed):
    M, N, K = 512, 19456, 384
    g = torch.Generator(device="cuda").manual_seed(seed)
    A = torch.randint(-40, 41, (M, K), generator=g, device="cuda").double()
    B = torch.randint(-40, 41, (N, K), generator=g, device="cuda").double()
    out = torch.zeros(N, M, device="cuda")
    work = torch.empty(8 * (M + N) * (K + 8) + 1024, dtype=torch.uint8, device="cuda")
    st = L.lib.tpt_tc_gemm_out(L.TPT_PREC_MIXED_BF16X3, M, N, K, C.c_void_p(A.data_ptr()), C.c_void_p(B.data_ptr()),
                               L.TPT_GEMM_OUT_F32, 1 << 30, 0, M, C.c_void_p(out.data_ptr()), None,
                               C.c_void_p(work.data_ptr()), C.c_void_p(torch.cuda.current_stream().cuda_stream),
                               256, 1, 0)
    assert st == L.TPT_OK
    torch.cuda.synchronize()
    return torch.equal(out.double(), B @ A.T)


@pytest.mark.parametrize("rank", [0, 1])
def test_a_pair_that_stops_early_waits_for_its_copies(rank):
    work = torch.zeros(1 << 27, dtype=torch.uint8, device="cuda")
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    for i in range(3):
        st = L.lib.tpt_test_pair_timeout(1 << 11, rank, C.c_void_p(work.data_ptr()), work.numel(), stream)
        assert st == L.TPT_ERR_TIMEOUT, L.lib.tpt_status_string(st)
        assert _exact_product(i)
    bad = L.lib.tpt_test_pair_timeout(1 << 11, 2, C.c_void_p(work.data_ptr()), work.numel(), stream)
    assert bad == L.TPT_ERR_INVALID_ARG
