"""GPU: the fixed-point state expansion of large single distributions against
the oracle at the bounds of its register lists (4, 8, 12 photons) and beside them, for bunched
inputs, matrices that are not unitary and ranges; and its FP64 form, which
matrices with entries of very different size, or none that is finite, take,
against the batched FP64 expansion.  Tolerances: 1e-10 relative with the RMS
floor, TVD 1e-12 (53 bits of the typical amplitude per level); the FP64 forms
differ by rounding alone, n additions of 2^-53 each: 1e-13."""
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


@pytest.mark.parametrize("m,n,t,form", [
    (998, 2, None, "haar"), (58, 4, [1] * 4, "haar"), (34, 5, [2, 1, 1, 1], "gauss"), (24, 6, [3, 0, 2, 1], "haar"),
    (20, 7, None, "scaled"), (16, 8, None, "gauss"), (14, 9, [9], "haar"), (12, 10, None, "haar"),
    (10, 12, [4] + [1] * 8, "haar"), (10, 12, [12], "haar"), (11, 11, [4, 4, 3], "scaled")])
def test_matches_oracle(pcv, m, n, t, form):
    full = np.zeros(m, np.uint8)
    if t is None:
        full[:min(n, m)] = 1
        full[0] += n - int(full.sum())
    else:
        full[:len(t)] = t
    U = pin.haar_unitary(m, 9700 + m)
    if form == "scaled":                       # columns of different norms
        U = U * 2.0 ** np.linspace(-7.3, 6.1, m)[None, :]
    elif form == "gauss":
        g = np.random.default_rng(97)
        U = g.standard_normal((m, m)) + 1j * g.standard_normal((m, m))
    p, a = pcv.distribution(dev(U), full)
    N = math.comb(m + n - 1, n)
    lo, hi = N // 3, N // 3 + 70000
    q, b = pcv.distribution_range(dev(U), full, lo, min(hi, N))
    torch.cuda.synchronize()
    assert torch.equal(q, p[lo:hi]) and torch.equal(b, a[lo:hi])
    if n <= 10:
        pick = slice(None)
        p_ref, a_ref = oracle.distribution(U, full)
    else:                                      # plain double Ryser is 1.3e-10 off double-double's here
        pick = slice(None, None, 8)
        a_ref = oracle.amplitudes(U, full, oracle.enumerate_outputs(m, n)[pick], method="ryser_dd")
        p_ref = np.abs(a_ref) ** 2
    p, a = p.cpu().numpy()[pick], a.cpu().numpy()[pick]
    rms = math.sqrt(np.mean(p_ref))
    assert np.max(np.abs(a - a_ref) / np.maximum(np.abs(a_ref), rms)) <= 1e-10
    assert oracle.tvd(p / p_ref.sum(), p_ref / p_ref.sum()) <= 1e-12


@pytest.mark.parametrize("form", ["coupling", "zero_column", "nan", "inf", "huge"])
def test_fp64_form(pcv, form):
    m, n = 19, 7
    t = pin.single_photon_input(m, n)
    U = pin.haar_unitary(m, 9790)
    if form == "coupling":                     # weakly coupled modes: outputs down to 1e-60
        U = np.eye(m) + 1e-9 * U
    elif form == "zero_column":
        U[:, 2] = 0
    elif form == "huge":
        U[:, 1] *= 2.0 ** 60
    else:
        U[3, 4] = np.nan if form == "nan" else np.inf
    p, a = pcv.distribution(dev(U), t)
    P, A = pcv.distribution_batched(dev(np.stack([U, U])), t)
    torch.cuda.synchronize()
    for x, y in ((p, P[0]), (torch.view_as_real(a), torch.view_as_real(A[0]))):
        assert torch.equal(torch.isnan(x), torch.isnan(y))
        x, y = torch.nan_to_num(x, nan=0.0), torch.nan_to_num(y, nan=0.0)
        assert torch.allclose(x, y, rtol=1e-13, atol=0.0)
