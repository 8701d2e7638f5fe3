"""GPU: forms that a size or a workspace chooses, each shown to be the one that
ran: the distribution's adjoint by minors in a workspace too small for the
levels (launch counts differ), against the reverse expansion (1e-10 of the
gradient's largest entry); and the sampler at the photon numbers where its
levels turn to fixed point (10) and take 256 threads (13), also for a matrix
near the identity, draw for draw against the numpy restatement."""
import math

import numpy as np
import pytest
import torch

import pcv_inputs as pin
from test_gpu_sampler_levels import reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,B,t", [
    (1, 3, 2, [3]), (2, 1, 1, None), (5, 3, 3, None), (3, 9, 2, [4, 3, 2]), (33, 2, 2, None), (8, 6, 7, None)])
def test_adjoint_in_a_small_workspace_takes_the_minors(m, n, B, t):
    from paper_2204_00602_gb300 import _abi as abi
    t = pin.single_photon_input(m, n) if t is None else np.array(t, np.uint8)
    U = torch.from_numpy(np.stack([pin.haar_unitary(m, 9990 + b) for b in range(B)])).cuda()
    g = np.random.default_rng(9991)
    N = math.comb(m + n - 1, n)
    gamp = torch.from_numpy(g.standard_normal((B, N)) + 1j * g.standard_normal((B, N))).cuda()
    out, launches = [], []
    for nbytes in (abi.pcv_distribution_backward_workspace(B, m, n), abi.pcv_amplitudes_backward_workspace(B, m, n, 1)):
        ws, gU = torch.empty(nbytes, dtype=torch.uint8, device="cuda"), torch.empty_like(U)
        before = abi.pcv_launch_count()
        abi.pcv_distribution_backward(U, B, m, t, gamp, gU, ws, nbytes, torch.cuda.current_stream().cuda_stream)
        launches.append(abi.pcv_launch_count() - before)
        out.append(gU)
    assert launches[0] == 2 * n + 3            # count table, ranks, n - 1 levels, seed, n levels back, sums
    assert launches[1] != launches[0]
    assert (out[1] - out[0]).abs().max().item() <= 1e-10 * out[0].abs().max().item()


@pytest.mark.parametrize("m,n,count,form", [
    (21, 10, 37, "haar"), (10, 10, 50, "near_identity"), (50, 13, 17, "haar"), (16, 13, 21, "near_identity")])
def test_sampler_forms_draw_for_draw(m, n, count, form):
    import paper_2204_00602_gb300 as pcv
    t = pin.single_photon_input(m, n)
    U = pin.haar_unitary(m, 9992 + n)
    if form == "near_identity":
        w, v = np.linalg.eigh(U + U.conj().T)
        U = np.ascontiguousarray((v * np.exp(0.1j * w)) @ v.conj().T)
    perm, uni = pin.sampler_randomness(count, n, 9993)
    got = pcv.sample(torch.from_numpy(U).cuda(), t, torch.from_numpy(perm).cuda(), torch.from_numpy(uni).cuda())
    assert np.array_equal(got.cpu().numpy(), reference(U, t, perm, uni))
