"""GPU: exact sampling against a numpy restatement on the same random numbers
(sub-permanents by the expansion along the drawn rows): every photon number
where the kernel's thread groups change, odd mode counts, counts that do not
fill a block, bunched inputs.  The samples are equal: a draw could differ only
where a uniform number falls within rounding (1e-13) of a boundary."""
import itertools

import numpy as np
import pytest
import torch

import pcv_inputs as pin

pytestmark = pytest.mark.gpu


def reference(U, t, perm, uni):
    m = U.shape[0]
    cols = np.repeat(np.arange(m), t)
    count, n = perm.shape
    A = U[:, cols[perm]].transpose(1, 0, 2)                  # [count, m, n]
    order = sorted(range(m), key=lambda i: (i % 32, i // 32))   # the kernel's cumulative order
    f = {(): np.ones(count, complex)}
    occ = np.zeros((count, m), np.uint8)
    for k in range(1, n + 1):
        sub = np.stack([f[tuple(x for x in range(k) if x != l)] for l in range(k)], 1)
        w = np.abs(np.einsum("cml,cl->cm", A[:, :, :k], sub)) ** 2
        cum = np.cumsum(w[:, order], axis=1)
        pick = (cum <= (uni[:, k - 1] * cum[:, -1])[:, None]).sum(1)
        r = np.array(order)[np.minimum(pick, m - 1)]
        np.add.at(occ, (np.arange(count), r), 1)
        if k < n:
            row = A[np.arange(count), r]                     # [count, n]
            f = {S: sum(row[:, l] * f[tuple(x for x in S if x != l)] for l in S)
                 for S in itertools.combinations(range(n), k)}
    return occ


@pytest.mark.parametrize("m,n,count,t", [
    (1, 2, 3, [2]), (5, 1, 40, None), (7, 2, 65, None), (33, 8, 61, None), (20, 9, 35, None), (9, 11, 33, [3, 0, 2, 2, 1, 1, 1, 1, 0]),
    (41, 12, 21, None), (60, 14, 19, None), (128, 15, 9, None), (17, 16, 7, None)])
def test_matches_numpy_draw_for_draw(m, n, count, t):
    import paper_2204_00602_gb300 as pcv
    t = pin.single_photon_input(m, n) if t is None else np.array(t, np.uint8)
    U = pin.haar_unitary(m, 9700 + n)
    perm, uni = pin.sampler_randomness(count, n, 9701)
    got = pcv.sample(torch.from_numpy(U).cuda(), t, torch.from_numpy(perm).cuda(), torch.from_numpy(uni).cuda())
    assert np.array_equal(got.cpu().numpy(), reference(U, t, perm, uni))
