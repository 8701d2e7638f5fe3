"""GPU: the state expansion asked for by name (PCV_ALGO_SLOS) keeps every
output's own precision at sizes where the default choice may sum in fixed
point: matrices whose outputs span many orders of magnitude.  An output of n
photons is a sum of products with at most 2n roundings each and about m n
additions of like terms, so its error is below (2 n + m n) 2^-52 < 1e-13 of the
permanent of the magnitudes; oracle: the n! terms summed one by one.  The
default choice takes the same FP64 sums for such matrices (equal to rounding
with the batched form, which always does), and fixed point for others, where no
output comes out as zero and errors stay below 2^-48 of the largest amplitude (n
levels of a few units of 2^-53)."""
import numpy as np
import pytest
import torch

import oracle
import pcv_inputs as pin

pytestmark = pytest.mark.gpu

M, N = 19, 7                                    # 657,800 states in all


def matrix(form):
    U = pin.haar_unitary(M, 9950)
    if form == "rows":                          # modes of very different loss
        return 2.0 ** np.linspace(0, -17, M)[:, None] * U
    if form == "crossing":                      # weak beam splitters, zeros beside them
        U = np.eye(M, dtype=complex)
        for j in range(N):
            U[j, j] = U[N + j, N + j] = np.sqrt(1 - 2.0 ** -20)
            U[N + j, j], U[j, N + j] = 2.0 ** -10, -2.0 ** -10
        return U
    return np.eye(M) + float(form) * U          # weakly coupled modes


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("form", ["1e-3", "1e-4", "1e-5", "rows"])
def test_named_expansion_is_relative(form):
    import paper_2204_00602_gb300 as pcv
    U, t = matrix(form), pin.single_photon_input(M, N)
    _, a = pcv.distribution(dev(U), t, algo=pcv.PCV_ALGO_SLOS)
    a = a.cpu().numpy()
    outs = oracle.enumerate_outputs(M, N)
    pick = np.concatenate([np.arange(100), np.arange(len(outs) - 100, len(outs)),
                           np.random.default_rng(9951).choice(len(outs), 100, replace=False)])
    ref = oracle.amplitudes(U, t, outs[pick], method="leibniz")
    size = np.abs(oracle.amplitudes(np.abs(U).astype(complex), t, outs[pick], method="leibniz"))
    assert np.max(np.abs(a[pick] - ref) / size) <= 1e-13
    assert not (a == 0).any()


@pytest.mark.parametrize("form", ["1e-2", "1e-3", "1e-4", "rows", "crossing"])
def test_default_keeps_fp64_where_outputs_span_much(form):
    import paper_2204_00602_gb300 as pcv
    U, t = dev(matrix(form)), pin.single_photon_input(M, N)
    _, a = pcv.distribution(U, t)
    _, b = pcv.distribution_batched(torch.stack([U, U]), t)
    assert torch.allclose(torch.view_as_real(a), torch.view_as_real(b[0]), rtol=1e-13, atol=0)


@pytest.mark.parametrize("form", ["haar", "0.3"])
def test_default_takes_fixed_point_for_others(form):
    import paper_2204_00602_gb300 as pcv
    U = dev(pin.haar_unitary(M, 9952) if form == "haar" else matrix(form))
    t = pin.single_photon_input(M, N)
    _, a = pcv.distribution(U, t)
    _, b = pcv.distribution_batched(torch.stack([U, U]), t)
    assert not torch.equal(a, b[0])
    assert not (a == 0).any()
    assert (a - b[0]).abs().max().item() <= 2.0 ** -48 * b.abs().max().item()
