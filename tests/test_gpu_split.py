"""GPU: explicit outputs from two half expansions against the Glynn kernels
(n <= 12: 1e-10 relative with the RMS floor, n = 16: 1e-8): every lane count
and register bound, bunched outputs and inputs, wrong photon numbers, and the
many-unitaries form in shared memory."""
import math

import numpy as np
import pytest
import torch

import pcv_inputs as pin

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pcv():
    import paper_2204_00602_gb300 as pcv
    return pcv


def outputs(m, n, count, seed):
    o = pin.random_bunched_outputs(m, n, count, seed)
    o[0] = 0
    o[0, m - 1] = n                        # every photon in one mode
    o[-1] = pin.random_bunched_outputs(m, n + 1, 1, seed + 1)[0]     # another photon number: amplitude 0
    return o


@pytest.mark.parametrize("m,n,count,t", [
    (9, 4, 200_000, None), (20, 7, 9_000, None), (12, 8, 45_000, [2, 0, 1, 0, 0, 3, 0, 0, 1, 0, 0, 1]),
    (20, 10, 4_097, None), (14, 10, 39_001, None), (16, 11, 3_000, None), (13, 12, 40_001, None), (11, 16, 700, [2, 2, 2, 2, 2, 1, 1, 1, 1, 1, 1])])
def test_split_matches_glynn(pcv, m, n, count, t):
    t = pin.single_photon_input(m, n) if t is None else np.array(t, np.uint8)
    U = torch.from_numpy(pin.haar_unitary(m, 9500)).cuda()
    o = torch.from_numpy(outputs(m, n, count, 9501)).cuda()
    # the split form is what a full workspace gets: more than the Glynn kernel's own need
    assert pcv.abi.pcv_amplitudes_workspace(m, n, count) >= 2 * 2 * 16 * math.comb(m + (n + 1) // 2 - 1, (n + 1) // 2)
    a, p = pcv.amplitudes(U, t, o)
    ref, q = pcv.amplitudes(U, t, o, algo=pcv.PCV_ALGO_TILE)
    floor = 1 / math.sqrt(math.comb(m + n - 1, n))
    err = ((a - ref).abs() / ref.abs().clamp(min=floor)).max().item()
    assert err <= (1e-10 if n <= 12 else 1e-8)
    assert a[-1] == 0 and p[-1] == 0
    assert torch.allclose(p, q, rtol=0, atol=1e-10 * q.max().item())


def test_small_workspace_takes_the_glynn_kernel(pcv):
    m, n = 20, 10
    U = torch.from_numpy(pin.haar_unitary(m, 9510)).cuda()
    t = pin.single_photon_input(m, n)
    o = torch.from_numpy(outputs(m, n, 4096, 9511)).cuda()
    a, _ = pcv.amplitudes(U, t, o)
    amp, prob = torch.empty_like(a), torch.empty(4096, dtype=torch.float64, device="cuda")
    pcv.abi.pcv_amplitudes_ex(U, m, t, o, 4096, amp, prob, pcv.PCV_ALGO_AUTO, 0, None, 0,
                              torch.cuda.current_stream().cuda_stream)
    ref, _ = pcv.amplitudes(U, t, o, algo=pcv.PCV_ALGO_GROUP, param=32)
    assert torch.equal(amp, ref)
    assert (a - ref).abs().max().item() <= 1e-10 * ref.abs().max().item()


@pytest.mark.parametrize("m,n,B,count", [(3, 2, 5, 40), (6, 4, 3, 129), (12, 6, 7, 512), (12, 6, 400, 65), (9, 5, 1, 1000),
                                         (8, 7, 2, 300), (16, 8, 3, 200), (7, 10, 2, 257)])
def test_split_multi_matches_glynn(pcv, m, n, B, count):
    t = pin.single_photon_input(m, n) if n <= m else np.array([2, 2, 2, 1, 1, 1, 1], np.uint8)
    U = torch.from_numpy(np.stack([pin.haar_unitary(m, 9520 + b) for b in range(B)])).cuda()
    o = torch.from_numpy(outputs(m, n, count, 9521)).cuda()
    amp = torch.empty(B, count, dtype=torch.complex128, device="cuda")
    prob = torch.empty(B, count, dtype=torch.float64, device="cuda")
    pcv.abi.pcv_amplitudes_multi(U, B, m, t, o, count, amp, prob, torch.cuda.current_stream().cuda_stream)
    floor = 1 / math.sqrt(math.comb(m + n - 1, n))
    for b in sorted({0, B // 2, B - 1}):
        ref, q = pcv.amplitudes(U[b], t, o, algo=pcv.PCV_ALGO_TILE)
        assert ((amp[b] - ref).abs() / ref.abs().clamp(min=floor)).max().item() <= 1e-10
        assert torch.allclose(prob[b], q, rtol=0, atol=1e-10 * q.max().item())
