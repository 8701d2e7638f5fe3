"""GPU: the distribution's adjoint by the reverse state expansion against the
minors as Glynn sums (the same outputs given explicitly), which the oracle
pins: 1e-10 of the gradient's largest entry, as for the forward amplitudes."""
import math

import numpy as np
import pytest
import torch

import oracle
import pcv_inputs as pin

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,B,t", [
    (1, 3, 2, [3]), (2, 1, 1, None), (5, 3, 3, None), (9, 4, 5, [0, 2, 0, 1, 0, 0, 0, 1, 0]), (3, 9, 2, [4, 3, 2]),
    (33, 2, 2, None), (8, 6, 7, None), (10, 6, 150, None)])
def test_matches_the_minors(m, n, B, t):
    from paper_2204_00602_gb300 import _abi as abi
    from paper_2204_00602_gb300 import autograd as ag
    t = pin.single_photon_input(m, n) if t is None else np.array(t, np.uint8)
    N = math.comb(m + n - 1, n)
    U = torch.from_numpy(np.stack([pin.haar_unitary(m, 9300 + b) for b in range(B)])).cuda()
    g = np.random.default_rng(9301)
    gamp = torch.from_numpy(g.standard_normal((B, N)) + 1j * g.standard_normal((B, N))).cuda()
    got = ag.distribution_backward(U, t, gamp)
    assert torch.equal(got, ag.distribution_backward(U, t, gamp))
    outs = torch.from_numpy(oracle.enumerate_outputs(m, n)).cuda()
    ref = torch.empty_like(U)
    ws = torch.empty(abi.pcv_amplitudes_backward_workspace(B, m, n, N), dtype=torch.uint8, device="cuda")
    abi.pcv_amplitudes_backward_multi(U, B, m, t, outs, N, gamp, ref, ws, ws.numel(),
                                      torch.cuda.current_stream().cuda_stream)
    # a workspace too small for the levels takes the minors itself
    small = torch.empty_like(U)
    nb = 64 << 10
    plan = abi.pcv_amplitudes_backward_workspace(B, m, n, 1)
    ws2 = torch.empty(max(nb, plan), dtype=torch.uint8, device="cuda")
    abi.pcv_distribution_backward(U, B, m, t, gamp, small, ws2, ws2.numel(), torch.cuda.current_stream().cuda_stream)
    scale = ref.abs().max().item()
    assert (got - ref).abs().max().item() <= 1e-10 * scale
    assert (small - ref).abs().max().item() <= 1e-10 * scale
