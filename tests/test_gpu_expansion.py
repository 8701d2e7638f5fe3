"""GPU: the FP64 distribution by state expansion (batches, n > 10, ranges) at
the edges of its variants: register-list bounds (n = 4, 8, 16 and beyond, where
ranks are 64-bit), batches that do not fill a group of four, one mode, bunched
inputs.  Tolerances: 1e-10 relative with the RMS floor for n <= 12, 1e-8
beyond, TVD 1e-12 (the rounding of n additions of FP64 products is near
1e-15)."""
import math

import numpy as np
import pytest
import torch

import oracle
import pcv_inputs as pin

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pcv():
    import paper_2204_00602_gb300 as pcv
    return pcv


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def amp_err(a, ref, count):
    return np.max(np.abs(a - ref) / np.maximum(np.abs(ref), 1 / math.sqrt(count)))


@pytest.mark.parametrize("m,n,B,t", [
    (1, 4, 3, [4]), (2, 1, 1, None), (6, 4, 5, None), (7, 5, 4, [2, 0, 1, 1, 0, 0, 1]), (9, 8, 3, None),
    (5, 9, 6, [3, 2, 2, 1, 1]), (3, 16, 2, [6, 5, 5]), (2, 17, 2, [9, 8]), (12, 6, 52, None)])
def test_batched_distribution_matches_oracle(pcv, m, n, B, t):
    t = pin.single_photon_input(m, n) if t is None else np.array(t, np.uint8)
    U = np.stack([pin.haar_unitary(m, 9100 + b) for b in range(B)])
    prob, amp = pcv.distribution_batched(dev(U), t)
    torch.cuda.synchronize()
    for b in sorted({0, B // 2, B - 1}):
        if n <= 12:
            p_ref, a_ref = oracle.distribution(U[b], t)
        else:                              # plain double Ryser cancels too much for bunched inputs here
            a_ref = oracle.amplitudes(U[b], t, oracle.enumerate_outputs(m, n), method="ryser_dd")
            p_ref = np.abs(a_ref) ** 2
        assert amp_err(amp[b].cpu().numpy(), a_ref, len(p_ref)) <= (1e-10 if n <= 12 else 1e-8)
        assert oracle.tvd(prob[b].cpu().numpy(), p_ref) <= 1e-12


@pytest.mark.parametrize("want_amp", [True, False])
def test_more_than_ten_photons_whole_and_in_ranges(pcv, want_amp):
    m, n = 7, 12
    t = np.array([2, 2, 2, 2, 2, 1, 1], np.uint8)
    U = pin.haar_unitary(m, 9201)
    N = math.comb(m + n - 1, n)
    ws = torch.empty(pcv.abi.pcv_distribution_workspace(m, n), dtype=torch.uint8, device="cuda")
    assert pcv.abi.pcv_distribution_auto_algo(m, n, ws.numel()) == pcv.PCV_ALGO_FACTOR
    p, a = pcv.distribution(dev(U), t, want_amp=want_amp, ws=ws)
    f, g = pcv.distribution(dev(U), t, algo=pcv.PCV_ALGO_FACTOR)      # the factorised sum
    torch.cuda.synchronize()
    assert oracle.tvd(p.cpu().numpy(), f.cpu().numpy()) <= 1e-12
    if want_amp:
        assert amp_err(a.cpu().numpy(), g.cpu().numpy(), N) <= 1e-10
    cuts = [0, 1, N // 3, N // 3, N - 5, N]
    parts = [pcv.distribution_range(dev(U), t, lo, hi, want_amp=want_amp, ws=ws) for lo, hi in zip(cuts, cuts[1:])]
    assert torch.equal(torch.cat([x[0] for x in parts]), p)
    if want_amp:
        assert torch.equal(torch.cat([x[1] for x in parts]), a)
    assert pcv.distribution_status(ws) == pcv.abi.PCV_OK
