"""GPU: small full distributions (PCV_ALGO_AUTO's state expansion, every level in
one block, and the sizes just beyond one block) against the oracle: 1e-10
relative with the RMS floor, TVD 1e-12; ranges give the same bits."""
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


@pytest.mark.parametrize("m,n,t", [(1, 1, None), (1, 7, [7]), (2, 1, None), (6, 3, None), (24, 3, None), (140, 2, None),
                                   (10, 4, None), (9, 5, [0, 2, 0, 0, 3, 0, 0, 0, 0]), (11, 6, None), (4, 9, [3, 3, 2, 1]),
                                   (3, 12, [5, 4, 3]), (2, 10, [4, 6]), (7, 8, [2, 1, 1, 1, 1, 1, 1])])
@pytest.mark.parametrize("want_amp", [True, False])
def test_auto_matches_oracle_and_ranges(pcv, m, n, t, want_amp):
    t = pin.single_photon_input(m, n) if t is None else np.array(t, np.uint8)
    U = pin.haar_unitary(m, 9900 + n)
    Ud = torch.from_numpy(U).cuda()
    N = math.comb(m + n - 1, n)
    ws = torch.full((pcv.abi.pcv_distribution_workspace(m, n),), 255, dtype=torch.uint8, device="cuda")
    p, a = pcv.distribution(Ud, t, want_amp=want_amp, ws=ws)
    assert pcv.distribution_status(ws) == pcv.abi.PCV_OK
    # plain Ryser sums lose 2e-12 themselves at m=3 n=12: double-double ones
    a_ref = oracle.amplitudes(U, t, oracle.enumerate_outputs(m, n), method="ryser_dd")
    assert oracle.tvd(p.cpu().numpy(), np.abs(a_ref) ** 2) <= 1e-12
    if want_amp:
        err = np.abs(a.cpu().numpy() - a_ref) / np.maximum(np.abs(a_ref), 1 / math.sqrt(N))
        assert err.max() <= 1e-10
    cuts = sorted({0, N, N // 2, max(0, N - 1), min(1, N)})
    parts = [pcv.distribution_range(Ud, t, lo, hi, want_amp=want_amp, ws=ws) for lo, hi in zip(cuts, cuts[1:])]
    assert torch.equal(torch.cat([x[0] for x in parts]), p)
    if want_amp:
        assert torch.equal(torch.cat([x[1] for x in parts]), a)


@pytest.mark.parametrize("m,n,B", [(6, 3, 300), (5, 4, 1), (3, 7, 17)])
def test_batched_small(pcv, m, n, B):
    t = pin.single_photon_input(m, n) if n <= m else np.array([3, 2, 2], np.uint8)
    U = np.stack([pin.haar_unitary(m, 9950 + b % 5) for b in range(B)])
    p, a = pcv.distribution_batched(torch.from_numpy(U).cuda(), t)
    for b in sorted({0, B // 2, B - 1}):
        p_ref, a_ref = oracle.distribution(U[b], t)
        assert oracle.tvd(p[b].cpu().numpy(), p_ref) <= 1e-12
        assert np.abs(a[b].cpu().numpy() - a_ref).max() <= 1e-10
