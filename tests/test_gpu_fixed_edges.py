"""GPU: the fixed-point state expansion at its fewest photons (2 and 3: factors
consumed by a last level with its extra bits) and at the most modes that its
tables take (m n <= 2048), where a column of equal magnitudes leaves most bits
of a level unused.  The launch count tells that it is the form that ran.
Tolerance: an output is n! products with at most 2 n roundings of sqrt(2) 2^-53
of a typical product, here and in the reference, and the outputs' rms is
sqrt(n!) products: 8 n sqrt(n!) 2^-53 of the larger of output and rms for
columns of equal magnitudes, 64 times that for Haar columns, whose entries reach
several times the rms."""
import math

import numpy as np
import pytest
import torch

import oracle
import pcv_inputs as pin

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,form", [(1024, 2, "flat"), (682, 3, "flat"), (999, 2, "haar"), (145, 3, "haar")])
def test_few_photons_in_many_modes(m, n, form):
    import paper_2204_00602_gb300 as pcv
    if form == "flat":
        U = np.exp(2j * np.pi * np.random.default_rng(9980).random((m, m))) / math.sqrt(m)
    else:
        U = pin.haar_unitary(m, 9981)
    t = pin.single_photon_input(m, n)
    N = math.comb(m + n - 1, n)
    assert sum(math.comb(m + k - 1, k) for k in range(n + 1)) >= 500_000
    need = max(pcv.abi.pcv_distribution_workspace_min(m, n), pcv.abi.pcv_distribution_slos_workspace(1, m, n) + 256)
    ws, Ud = pcv.workspace(need, "cuda"), torch.from_numpy(U).cuda()
    lo = max(0, N // 2 - 200_000)
    hi = min(N, lo + 400_000)
    before = pcv.abi.pcv_launch_count()
    _, a = pcv.distribution_range(Ud, t, lo, hi, ws=ws)
    assert pcv.abi.pcv_launch_count() - before == n + 2       # count table, columns' norms, n levels
    pick = np.random.default_rng(9982).choice(hi - lo, 3000, replace=False)
    outs = np.stack([pcv.unrank(m, n, lo + int(i)) for i in pick])
    ref = oracle.amplitudes(U, t, outs, method="leibniz")
    rms = 1 / math.sqrt(N)
    err = np.abs(a.cpu().numpy()[pick] - ref) / np.maximum(np.abs(ref), rms)
    assert err.max() <= 8 * n * math.sqrt(math.factorial(n)) * 2.0 ** -53 * (1 if form == "flat" else 64)
