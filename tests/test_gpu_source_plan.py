"""GPU: the source model over all pure sets at once against one set at a time
(the path a smaller workspace takes): TVD <= 1e-12."""
import numpy as np
import pytest
import torch

import oracle
import pcv_inputs as pin

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,t,eta,V", [
    (1, 2, [2], 0.7, 0.5), (3, 1, None, 0.6, 0.2), (4, 3, None, 1.0, 0.8), (4, 3, [2, 0, 1, 0], 0.5, 0.0),
    (5, 4, None, 0.0, 0.5), (7, 5, [1, 0, 3, 0, 1, 0, 0], 0.9, 0.9), (3, 9, [4, 3, 2], 0.8, 0.7), (11, 5, None, 0.9, 1.0)])
def test_all_sets_at_once_matches_one_at_a_time(m, n, t, eta, V):
    import paper_2204_00602_gb300 as pcv
    from paper_2204_00602_gb300 import _abi as abi
    t = pin.single_photon_input(m, n) if t is None else np.array(t, np.uint8)
    U = torch.from_numpy(pin.haar_unitary(m, 9400)).cuda()
    p, off = pcv.source_distribution(U, t, eta, V)
    full = abi.pcv_distribution_source_workspace(m, t)
    lo, hi = 1, full                       # the smallest workspace the call accepts
    while lo < hi:
        mid = (lo + hi) // 2
        ws = torch.empty(mid, dtype=torch.uint8, device="cuda")
        try:
            pcv.source_distribution(U, t, eta, V, ws=ws)
            hi = mid
        except pcv.PcvError:
            lo = mid + 1
    q, _ = pcv.source_distribution(U, t, eta, V, ws=torch.empty(lo, dtype=torch.uint8, device="cuda"))
    torch.cuda.synchronize()
    assert abs(p.sum().item() - 1.0) <= 1e-12
    assert oracle.tvd(p.cpu().numpy(), q.cpu().numpy()) <= 1e-12
