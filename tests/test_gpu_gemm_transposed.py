"""GPU: the tcgen05 GEMM with operands read transposed in place: bit for bit
the product of the transposed copies (same sums, same order), at every tile
width, ragged edges, and K blocks that do not fill a stage."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(128, 128, 64), (8, 40, 24), (136, 72, 200), (1024, 288, 4096), (512, 1024, 1000),
                                   (4096, 1024, 512), (2000, 1016, 1024), (5000, 24, 72)])
@pytest.mark.parametrize("at,bt", [(0, 1), (1, 0), (1, 1)])
def test_matches_transposed_copies(M, N, K, at, bt):
    from paper_2204_00602_gb300 import _abi as abi
    g = torch.Generator(device="cuda").manual_seed(M + 3 * N + K)
    A = torch.randn(M, K, device="cuda", generator=g).to(torch.bfloat16)
    B = torch.randn(N, K, device="cuda", generator=g).to(torch.bfloat16)
    pre = torch.randn(M, N, device="cuda", generator=g)
    bias = torch.randn(N, device="cuda", generator=g)
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    At, Bt = A.t().contiguous(), B.t().contiguous()
    opA, lda = (At, M) if at else (A, K)
    opB, ldb = (Bt, N) if bt else (B, K)
    for mode in range(4):
        want_f, want_b = torch.zeros(M, N, device="cuda"), torch.zeros(M, N, device="cuda", dtype=torch.bfloat16)
        got_f, got_b = torch.full_like(want_f, float("nan")), torch.full_like(want_b, float("nan"))
        f = mode in (0, 1, 2)
        b = mode in (1, 3)
        args = lambda of, ob: (mode, bias if mode in (1, 2) else None, of if f else None, N, ob if b else None, N,
                               pre if mode == 3 else None, N, err, s)
        abi.pcv_gemm_bf16_tc(A, K, B, K, M, N, K, *args(want_f, want_b))
        abi.pcv_gemm_bf16_tc_t(opA, lda, at, opB, ldb, bt, M, N, K, *args(got_f, got_b))
        torch.cuda.synchronize()
        assert err.item() == 0
        if f:
            assert torch.equal(got_f, want_f)
        if b:
            assert torch.equal(got_b, want_b)
        if mode == 0:
            ref = A.double() @ B.double().t()
            bound = K * 2.0 ** -23 * (A.double().abs() @ B.double().abs().t())
            assert ((got_f.double() - ref).abs() <= bound).all()
