"""GPU: the tile kernel's integer-pipe products: split sequences, many modes,
every tile shape, rows of very different scales, exact zeros and non-finite
entries, against the plain FP64 Glynn kernels (1e-10 relative with the RMS
floor for n <= 12, 1e-8 beyond; for scaled rows relative to each row's scale)."""
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


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def plain(pcv, U, t, o, n):
    return pcv.amplitudes(U, t, o, algo=pcv.PCV_ALGO_BLOCK, param=1)[0] if n > 12 else \
        pcv.amplitudes(U, t, o, algo=pcv.PCV_ALGO_GROUP, param=min(32, 1 << (n - 1)))[0]


def rel(a, ref, floor):
    return ((a - ref).abs() / ref.abs().clamp(min=floor)).max().item()


@pytest.mark.parametrize("m,n,count", [(130, 9, 20_000), (300, 12, 1_001), (324, 14, 257), (225, 15, 33), (400, 17, 40),
                                       (1024, 13, 300), (64, 13, 95), (40, 14, 2_000)])
def test_auto_split_sequences(pcv, m, n, count):
    U, t = dev(pin.haar_unitary(m, 9800 + n)), pin.single_photon_input(m, n)
    o = dev(pin.random_outputs(m, n, count, 9801))
    a, p = pcv.amplitudes(U, t, o)
    ref = plain(pcv, U, t, o, n)
    assert rel(a, ref, 1 / math.sqrt(math.comb(m + n - 1, n))) <= (1e-10 if n <= 12 else 1e-8)
    assert torch.allclose(p, a.real ** 2 + a.imag ** 2, rtol=1e-14, atol=0)
    assert torch.equal(a, pcv.amplitudes(U, t, o)[0])


@pytest.mark.parametrize("n", range(1, 13))
@pytest.mark.parametrize("count", [1, 33, 65, 300])
def test_every_shape(pcv, n, count):
    m = 11
    t = np.zeros(m, np.uint8)
    np.add.at(t, np.random.default_rng(n).integers(0, m, n), 1)
    U = dev(pin.haar_unitary(m, 9810 + n))
    o = dev(pin.random_bunched_outputs(m, n, count, 9811))
    a, _ = pcv.amplitudes(U, t, o, algo=pcv.PCV_ALGO_TILE)
    assert rel(a, plain(pcv, U, t, o, n), 1 / math.sqrt(math.comb(m + n - 1, n))) <= 1e-10


def test_scaled_rows_zeros_and_non_finite(pcv):
    m, n, count = 16, 8, 500
    U0, t = pin.haar_unitary(m, 9820), pin.single_photon_input(m, n)
    o = pin.random_outputs(m, n, count, 9821)
    scale = 10.0 ** np.random.default_rng(9822).integers(-30, 30, m)
    a, _ = pcv.amplitudes(dev(U0 * scale[:, None]), t, dev(o), algo=pcv.PCV_ALGO_TILE)
    ref = plain(pcv, dev(U0), t, dev(o), n)
    s = dev(np.prod(np.where(o > 0, scale[None, :], 1.0), axis=1))
    assert rel(a / s, ref, 1 / math.sqrt(math.comb(m + n - 1, n))) <= 1e-10
    # a zero row, a row with one entry, tiny entries (below the normal range once squared)
    U1 = U0.copy()
    U1[3] = 0
    U1[4, 1:] = 0
    U1[5] *= 1e-290
    a, _ = pcv.amplitudes(dev(U1), t, dev(o), algo=pcv.PCV_ALGO_TILE)
    ref = plain(pcv, dev(U1), t, dev(o), n)
    k = o[:, 3] > 0
    assert (a[dev(k)] == 0).all()
    five = dev(o[:, 5] > 0)
    assert rel(a[~five], ref[~five], 1e-4) <= 1e-10
    assert rel(a[five] * 1e290, ref[five] * 1e290, 1e-4) <= 1e-10
    # non-finite entries reach exactly the outputs that use their row
    U2 = U0.copy()
    U2[7, 2] = np.inf
    U2[9, 0] = np.nan
    a, p = pcv.amplitudes(dev(U2), t, dev(o), algo=pcv.PCV_ALGO_TILE)
    hit = dev((o[:, 7] > 0) | (o[:, 9] > 0))
    assert torch.isnan(p[hit]).all() and torch.isfinite(p[~hit]).all()
    assert torch.equal(a[~hit], pcv.amplitudes(dev(U0), t, dev(o), algo=pcv.PCV_ALGO_TILE)[0][~hit])


def test_batched_split_and_whole_sequences(pcv):
    """Few large circuits among many small ones: split over blocks with the
    full workspace, whole tiles with the least workspace the call accepts."""
    g = np.random.default_rng(9830)
    circs = []
    for c in range(12):
        n = [15, 14, 3, 4, 5, 6, 13, 2, 1, 9, 7, 11][c]
        m = int(g.integers(n, 40))
        circs.append((dev(pin.haar_unitary(m, 9831 + c)), pin.single_photon_input(m, n),
                      dev(pin.random_outputs(m, n, [300, 70, 5, 33, 1, 129, 31, 64, 7, 260, 8, 90][c], 9850 + c))))
    plan = pcv.BatchPlan(circs)
    amps = [a.clone() for a in plan.run()[0]]
    lo, hi = 1, plan.ws.numel()
    full = plan.ws
    while lo < hi:
        mid = (lo + hi) // 2
        plan.ws = full[:mid]
        try:
            plan.run()
            hi = mid
        except pcv.PcvError:
            lo = mid + 1
    plan.ws = full[:lo]
    whole, _ = plan.run()
    torch.cuda.synchronize()
    assert lo < full.numel()
    for (U, t, o), a, w in zip(circs, amps, whole):
        m, n = U.shape[0], int(t.sum())
        floor = 1 / math.sqrt(math.comb(m + n - 1, n))
        ref = plain(pcv, U, t, o, n)
        tol = 1e-10 if n <= 12 else 1e-8
        assert rel(a, ref, floor) <= tol and rel(w, ref, floor) <= tol
