"""GPU: the surrogate's fused elementwise kernels.  Features and logarithms from
tables: as floats within one unit of the correctly rounded value (their FP64
error is below 1e-15), bf16 features equal; several tensors per launch: the
same bits as one tensor at a time, aligned or not."""
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


@pytest.mark.parametrize("B,P,ldx,span", [(1, 1, 3, 7.0), (5, 132, 288, 6.3), (300, 7, 15, -50.0), (64, 132, 265, 9e5),
                                          (3, 20, 48, 1e12)])
def test_features(abi, B, P, ldx, span):
    ph = torch.from_numpy(np.random.default_rng(P).uniform(0, span, (B, P)) if span > 0 else
                          np.random.default_rng(P).uniform(span, -span, (B, P))).cuda()
    ph[0, 0] = 0.0
    X = torch.full((B, ldx), 9.0, dtype=torch.bfloat16, device="cuda")
    abi.pcv_phase_features(ph, B, P, X, ldx, S())
    want = torch.zeros(B, ldx, dtype=torch.bfloat16, device="cuda")
    want[:, :P] = ph.sin().float().to(torch.bfloat16)
    want[:, P:2 * P] = ph.cos().float().to(torch.bfloat16)
    want[:, 2 * P] = 1
    assert torch.equal(X, want)


def test_log(abi):
    g = np.random.default_rng(1)
    x = np.concatenate([10.0 ** g.uniform(-300, 300, 5000), g.uniform(0, 2, 5000), 1 + g.uniform(-1e-6, 1e-6, 500),
                        1 + 10.0 ** -g.uniform(1, 15, 500), [1.0, 0.0, 5e-324, 1e-310, np.inf, -1.0, np.nan, 2.0, 0.5,
                                                             np.nextafter(1, 0), np.nextafter(2, 0), 1.7e308]])
    out = torch.empty(len(x), dtype=torch.float32, device="cuda")
    abi.pcv_log_f64_to_f32(torch.from_numpy(x).cuda(), len(x), out, S())
    with np.errstate(all="ignore"):
        want = np.log(x)
    got = out.cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(want))
    fin = np.isfinite(want)
    assert np.array_equal(got[~fin & ~np.isnan(want)], want[~fin & ~np.isnan(want)].astype(np.float32))
    assert np.all(np.abs(got[fin].astype(np.float64) - want[fin]) <= 2.0 ** -24 * 1.01 * np.abs(want[fin]) + 1e-45)


def test_several_tensors_per_launch(abi):
    g = torch.Generator(device="cuda").manual_seed(3)
    sizes = [1, 3, 1024, 1025, 4096 * 3 + 2, 7, 100, 5, 1 << 18, 2, 9, 11, 12, 13, 14, 15, 16, 17]
    base = [torch.randn(4, n + 1, device="cuda", generator=g) for n in sizes]
    one, many = [], []
    for dst in (one, many):
        for j, b in enumerate(base):
            w, m, v, gr = (b[r].clone()[j % 2:j % 2 + sizes[j]] for r in range(4))       # odd jobs misaligned
            dst.append((w, m, v.abs(), gr, torch.zeros(sizes[j] + 1, device="cuda", dtype=torch.bfloat16)[j % 2:][:sizes[j]]
                        if j % 3 else None))
    for w, m, v, gr, wb in one:
        abi.pcv_adam(w, m, v, gr, w.numel(), 1e-3, 0.9, 0.999, 1e-8, 4, wb, S())
    abi.pcv_adam_multi(many, 1e-3, 0.9, 0.999, 1e-8, 4, S())
    for a, b in zip(one, many):
        for x, y in zip(a, b):
            assert x is None or torch.equal(x, y)
    w, m, v, gr, wb = many[8]
    m2 = 0.9 * base[8][1][:sizes[8]].double() + 0.1 * gr.double()
    v2 = 0.999 * base[8][2][:sizes[8]].abs().double() + 0.001 * gr.double() ** 2
    ref = base[8][0][:sizes[8]].double() - 1e-3 * (m2 / (1 - 0.9 ** 4)) / ((v2 / (1 - 0.999 ** 4)).sqrt() + 1e-8)
    # the bias correction 1 - 0.999^4 = 0.004 is formed in float: 2^-24 / 0.004 relative
    assert (w.double() - ref).abs().max().item() <= 2e-6
    mats = [(torch.randn(M, ld, device="cuda", generator=g).to(torch.bfloat16), M, N, ld) for M, N, ld in
            [(1, 1, 1), (4096, 1024, 1024), (33, 7, 9), (256, 512, 600), (2049, 40, 40)]]
    sums = [torch.empty(N, device="cuda") for _, _, N, _ in mats]
    abi.pcv_colsum_bf16_multi([(d, M, N, ld, s) for (d, M, N, ld), s in zip(mats, sums)], S())
    for (d, M, N, ld), s in zip(mats, sums):
        single = torch.empty(N, device="cuda")
        abi.pcv_colsum_bf16(d, M, N, ld, single, S())
        assert torch.equal(s, single)
        want = d[:, :N].double().sum(0)
        assert ((s.double() - want).abs() <= M * 2.0 ** -23 * d[:, :N].double().abs().sum(0) + 1e-30).all()
