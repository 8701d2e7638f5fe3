"""GPU: mesh forward and reverse sweep column by column, at the sizes where a
column's MZIs leave threads over or need several passes (odd m, the largest m),
against the mesh written in torch with its autograd.  Tolerance: m column steps
of a unitary at FP64 rounding, 64 x 16 x 1.1e-16 < 2e-13, gradients 1e-11 of
their largest entry."""
import numpy as np
import pytest
import torch

import pcv_inputs as pin

pytestmark = pytest.mark.gpu


def torch_mesh(ph, m):
    rows = list(torch.eye(m, dtype=torch.complex128, device=ph.device).expand(ph.shape[0], m, m).unbind(1))
    q = 0
    for c in range(m):
        for k in range(c % 2, m - 1, 2):
            e, f = torch.exp(1j * ph[:, 2 * q])[:, None], torch.exp(1j * ph[:, 2 * q + 1])[:, None]
            u0, u1 = rows[k], rows[k + 1]
            rows[k] = 0.5 * ((e - 1) * u0 + 1j * (e + 1) * u1)
            rows[k + 1] = 0.5 * f * (1j * (e + 1) * u0 + (1 - e) * u1)
            q += 1
    return torch.stack(rows, 1)


@pytest.mark.parametrize("m,B", [(2, 1), (3, 4), (7, 3), (12, 65), (23, 2), (64, 2)])
def test_forward_and_backward(m, B):
    from paper_2204_00602_gb300 import autograd as ag
    ph = torch.from_numpy(pin.mesh_phases(B, m * (m - 1), 9600 + m)).cuda()
    U = ag.mesh_unitary(ph, m)
    p = ph.clone().requires_grad_(True)
    ref = torch_mesh(p, m)
    assert (U - ref).abs().max().item() <= 2e-13
    g = np.random.default_rng(9601)
    G = torch.from_numpy(g.standard_normal((B, m, m)) + 1j * g.standard_normal((B, m, m))).cuda()
    got = ag.mesh_backward(ph, U, G)
    # real loss with dL/dRe U + i dL/dIm U = G
    (ref.real * G.real + ref.imag * G.imag).sum().backward()
    assert (got - p.grad).abs().max().item() <= 1e-11 * p.grad.abs().max().item()
