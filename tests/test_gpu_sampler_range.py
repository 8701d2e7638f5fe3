"""GPU: exact sampling of matrices whose sub-permanents differ by many orders of
magnitude, against the same numpy expansion: inputs of very different loss
(columns scaled by up to 2^-29), weak couplings.  The uniform numbers are taken
from the middle of a mode's interval, the mode drawn among all with a weight of
1e-9 of the step's or more, so rare outcomes come up as often as others and the
samples are equal unless a weight is off by about its own size."""
import itertools

import numpy as np
import pytest
import torch

import pcv_inputs as pin

pytestmark = pytest.mark.gpu


def steered(U, cols, perm, g):
    """Uniforms and the samples that they lead to."""
    m, (count, n) = U.shape[0], perm.shape
    order = np.array(sorted(range(m), key=lambda i: (i % 32, i // 32)))     # the kernel's cumulative order
    A = U[:, cols[perm]].transpose(1, 0, 2)                  # [count, m, n]
    f = {(): np.ones(count, complex)}
    occ, uni, at = np.zeros((count, m), np.uint8), np.empty((count, n)), np.arange(count)
    for k in range(1, n + 1):
        sub = np.stack([f[tuple(x for x in range(k) if x != l)] for l in range(k)], 1)
        w = np.abs(np.einsum("cml,cl->cm", A[:, :, :k], sub))[:, order] ** 2
        w /= w.sum(1, keepdims=True)
        pick = np.argmax((w > 1e-9) * g.random((count, m)), axis=1)
        uni[:, k - 1] = np.cumsum(w, axis=1)[at, pick] - w[at, pick] / 2
        r = order[pick]
        np.add.at(occ, (at, r), 1)
        if k < n:
            row = A[at, r]
            row = row / np.abs(row).max(1, keepdims=True)    # the scale of a row cancels
            f = {S: sum(row[:, l] * f[tuple(x for x in S if x != l)] for l in S)
                 for S in itertools.combinations(range(n), k)}
    return uni, occ


@pytest.mark.parametrize("form", ["loss", "coupling1e-2", "coupling1e-4"])
@pytest.mark.parametrize("m,n,count", [(20, 10, 70), (23, 11, 33), (20, 12, 33), (18, 13, 17), (33, 14, 9), (16, 15, 5)])
def test_samples_of_wide_ranges(m, n, count, form):
    import paper_2204_00602_gb300 as pcv
    g = np.random.default_rng(9960 + n)
    U = pin.haar_unitary(m, 9961 + n)
    if form == "loss":
        U = U * np.exp2(-g.integers(0, 30, m).astype(float))
    else:
        w, v = np.linalg.eigh(U + U.conj().T)
        U = (v * np.exp(1j * float(form[8:]) * w)) @ v.conj().T
    t = pin.single_photon_input(m, n)
    perm, _ = pin.sampler_randomness(count, n, 9962)
    uni, want = steered(U, np.flatnonzero(t), perm, g)
    got = pcv.sample(torch.from_numpy(np.ascontiguousarray(U)).cuda(), t, torch.from_numpy(perm).cuda(), torch.from_numpy(uni).cuda())
    assert np.array_equal(got.cpu().numpy(), want)


def test_rows_that_are_not_finite():
    """A NaN in one input column: the samples are those of the photons before it, then mode 0."""
    import paper_2204_00602_gb300 as pcv
    m, n = 20, 10
    U = pin.haar_unitary(m, 9970)
    t = pin.single_photon_input(m, n)
    perm = np.tile(np.arange(n, dtype=np.uint8), (40, 1))
    uni, want = steered(U, np.flatnonzero(t), perm[:, :4], np.random.default_rng(9971))
    U = U.copy()
    U[:, 4] = np.nan
    uni = np.concatenate([uni, np.full((40, n - 4), 0.5)], 1)
    want[:, 0] += n - 4
    got = pcv.sample(torch.from_numpy(U).cuda(), t, torch.from_numpy(perm).cuda(), torch.from_numpy(uni).cuda())
    assert np.array_equal(got.cpu().numpy(), want)
