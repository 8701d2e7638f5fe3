"""GPU: explicit amplitudes of few outputs with 13 and more photons (m <= 128):
the default choice is no slower than the block kernel, which has the whole GPU
for a call of any size, and no less accurate.  Time: within a factor of two
(fewest of several timings; a permanent on a single warp took 5 to 35 times as
long).  Accuracy: rms error against double-double Ryser within 1.5 times the
block kernel's (both round every term to double; sums of weighted terms, each
standing for several sign vectors, were 3 to 5 times worse)."""
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


def collision_free(m, n, count, seed):
    g = np.random.default_rng(seed)
    o = np.zeros((count, m), np.uint8)
    o[np.arange(count)[:, None], np.argsort(g.random((count, m)), axis=1)[:, :n]] = 1
    return o


def block_parts(n, count):
    parts = 1
    while parts * 2 * 256 <= 1 << (n - 1) and count * parts < 152 * 8:
        parts *= 2
    return parts


def least_ms(fn):
    fn()
    best = float("inf")
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        fn()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("m,n,count,bunched", [
    (24, 17, 7, True), (40, 16, 8, True), (24, 18, 33, False), (40, 18, 65, False), (24, 15, 257, False),
    (128, 17, 16, True), (24, 14, 33, False), (128, 20, 7, True), (24, 20, 1, False)])
def test_no_slower_than_the_block_kernel(pcv, m, n, count, bunched):
    U, t = dev(pin.haar_unitary(m, 9900 + n)), pin.single_photon_input(m, n)
    o = dev(pin.random_bunched_outputs(m, n, count, 9901) if bunched else collision_free(m, n, count, 9901))
    auto = least_ms(lambda: pcv.amplitudes(U, t, o))
    block = least_ms(lambda: pcv.amplitudes(U, t, o, algo=pcv.PCV_ALGO_BLOCK, param=block_parts(n, count)))
    assert auto <= 2 * block


@pytest.mark.parametrize("m,n,count", [(15, 15, 64), (24, 17, 32), (17, 17, 33), (40, 16, 31)])
def test_no_less_accurate_than_the_block_kernel(pcv, m, n, count):
    U, t = pin.haar_unitary(m, 9910 + n), pin.single_photon_input(m, n)
    o = pin.random_bunched_outputs(m, n, count, 9911)
    ref = oracle.amplitudes(U, t, o, method="ryser_dd")
    rms = {}
    for name, algo, param in (("auto", pcv.PCV_ALGO_AUTO, 0), ("block", pcv.PCV_ALGO_BLOCK, block_parts(n, count))):
        a = pcv.amplitudes(dev(U), t, dev(o), algo=algo, param=param)[0].cpu().numpy()
        rms[name] = np.sqrt(np.mean(np.abs(a - ref) ** 2))
    assert rms["auto"] <= 1.5 * rms["block"]
