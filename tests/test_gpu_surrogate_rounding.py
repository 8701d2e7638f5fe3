"""GPU: the surrogate's sines, cosines and logarithms are the FP64 functions'
values rounded to floats, bit for bit, also where the FP64 value lies beside the
middle between two floats: there a table's larger FP64 error would show."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def abi():
    from paper_2204_00602_gb300 import _abi
    return _abi


def S():
    return torch.cuda.current_stream().cuda_stream


def middles(lo, hi, count, bits, seed):
    """Doubles in the middle between two floats; with bits = 16 between two of which one
    is itself the middle between two bf16 values, so the bf16 result turns there too."""
    f = np.random.default_rng(seed).uniform(lo, hi, count).astype(np.float32).view(np.int32)
    if bits:
        f = (f & ~0xFFFF) | np.where(np.arange(count) % 2, 0x7FFF, 0x8000).astype(np.int32)
    return (f.view(np.float32).astype(np.float64) + (f + 1).view(np.float32).astype(np.float64)) / 2


@pytest.mark.parametrize("lo,hi", [(0.0101, 0.02), (0.02, 0.7), (0.7, 30.0), (30.0, 700.0)])
def test_log_beside_the_middle_of_two_floats(abi, lo, hi):
    y = middles(lo, hi, 200_000, 0, 1)
    x = np.exp(np.concatenate([y, -y]))
    x = torch.from_numpy(np.concatenate([x, np.nextafter(x, 0), np.nextafter(x, np.inf)])).cuda()
    out = torch.empty(len(x), dtype=torch.float32, device="cuda")
    abi.pcv_log_f64_to_f32(x, len(x), out, S())
    assert torch.equal(out, x.log().float())


@pytest.mark.parametrize("turns", [0, 1, -2, 150])
def test_features_beside_the_middle_of_two_floats(abi, turns):
    v = middles(0.05, 0.999, 200_000, 16, 2)
    x = np.concatenate([np.arcsin(v), np.arccos(v), np.pi - np.arcsin(v)]) + 2 * np.pi * turns
    x = np.concatenate([x, np.nextafter(x, -9e9), np.nextafter(x, 9e9)])
    P = 50
    ph = torch.from_numpy(x).cuda().reshape(-1, P)
    X = torch.empty(len(ph), 2 * P + 1, dtype=torch.bfloat16, device="cuda")
    abi.pcv_phase_features(ph, len(ph), P, X, 2 * P + 1, S())
    assert torch.equal(X[:, :P], ph.sin().float().to(torch.bfloat16))
    assert torch.equal(X[:, P:2 * P], ph.cos().float().to(torch.bfloat16))
