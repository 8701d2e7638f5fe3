"""GPU: the state expansion asked for by name (PCV_ALGO_SLOS) keeps every
output's own precision at sizes where the default choice may sum in fixed
point: matrices whose outputs span many orders of magnitude.  An output of n
photons is a sum of products with at most 2n roundings each and about m n
additions of like terms, so its error is below (2 n + m n) 2^-52 < 1e-13 of the
permanent of the magnitudes; oracle: the n! terms summed one by one."""
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
