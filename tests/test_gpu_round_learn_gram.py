"""The rounding-learning step with many calibration rows, where the gradient is E (A^T A) instead of (A E^T)^T A: on both
sides of the rule that chooses it."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2408_06995_b200 as fpq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mean", [0.0, 2.0])
@pytest.mark.parametrize("M,N,K", [(128, 100, 64), (127, 100, 64), (8, 3, 4), (300, 200, 132), (640, 960, 320), (639, 960, 320),
                                   (2048, 700, 256), (1024, 2100, 256), (1700, 260, 204)])
def test_matches_the_oracle_at_fp32_accuracy(M, N, K, mean):
    rng = np.random.default_rng(M + N + K)
    w = (rng.standard_normal((N, K)) * 0.02).astype(np.float32)
    a = (rng.standard_normal((M, K)) + mean).astype(np.float32)
    scale = np.array([O.scale_from_max(v, O.E2M1) for v in np.abs(w).max(axis=1)], dtype=np.float32)
    alpha = (rng.standard_normal((N, K)) * 1.5).astype(np.float32)
    d = [torch.from_numpy(v).cuda() for v in (w, scale, alpha, a)]
    grad, loss = fpq.fpq_round_learn_step(d[0], d[1], fpq.E2M1, d[2], d[3], 0.0)
    assert fpq.fpq_read_status() == fpq.OK
    r = O.round_learn_step(w, scale, O.E2M1, alpha, a, 0.0)
    # products and their operands' splits leave out less than 2^-19 of a term, sums are FP32 in short chunks: the bounds
    # of test_gpu_round_learn.py's accuracy test, relative to the terms that are added here, |E| (|A|^T |A|)
    assert float(loss[0]) == pytest.approx(r["mse"], rel=1e-5)
    assert float(loss[1]) == pytest.approx(r["reg"], rel=1e-6)
    e = np.abs(r["wq"] - w.astype(np.float64))
    dwq = O.soft_weight(w, scale, O.E2M1, alpha)[1]
    terms = 2.0 / (M * N) * (e @ (np.abs(a.astype(np.float64)).T @ np.abs(a.astype(np.float64)))) * np.abs(dwq)
    err = np.abs(grad.cpu().numpy().astype(np.float64) - r["grad"])
    assert np.all(err <= 5e-6 * terms + 4.0 * np.spacing(np.abs(r["grad"]).astype(np.float32)).astype(np.float64) + 1e-16)
    assert np.linalg.norm(err) <= 1e-5 * np.linalg.norm(r["grad"])


def test_repeated_calls_agree_and_descend():
    g = torch.Generator(device="cuda").manual_seed(2)
    w = torch.randn(200, 128, generator=g, device="cuda") * 0.02
    a = torch.randn(1000, 128, generator=g, device="cuda") + 0.5
    scale = (w.abs().amax(dim=1) / 6).contiguous()
    alpha = torch.randn(200, 128, generator=g, device="cuda") * 0.1
    g1, l1 = fpq.fpq_round_learn_step(w, scale, fpq.E2M1, alpha, a, 1e-6)
    g2, _ = fpq.fpq_round_learn_step(w, scale, fpq.E2M1, alpha, a, 1e-6)
    assert torch.equal(g1, g2)
    first = float(l1[0])
    for _ in range(20):
        _, loss = fpq.fpq_round_learn_step(w, scale, fpq.E2M1, alpha, a, 0.0, lr=1e5)
    assert 0.0 < float(loss[0]) < first


# the product with E in tiles of 32, 40, 48 and 64 rows, several rounds of them, the last one ragged in rows and columns; one
# and many slices of A^T A; the direct form; step sizes and decisions that are not 16-byte aligned
@pytest.mark.parametrize("M,N,K,lr", [(700, 33, 68, 0.0), (700, 961, 316, 1e4), (700, 1700, 256, 0.0), (600, 2350, 252, 1e4),
                                      (200, 9500, 60, 0.0), (1100, 1500, 400, 0.0), (1100, 600, 316, 0.0), (1200, 700, 580, 1e4)])
@pytest.mark.parametrize("offset", [0, 1])
def test_gradient_tiles(M, N, K, lr, offset):
    gen = torch.Generator(device="cuda").manual_seed(N + K)
    w = torch.randn(N, K, generator=gen, device="cuda") * 0.02
    a = torch.randn(M, K, generator=gen, device="cuda") + 0.2
    scale = (w.abs().amax(dim=1) / 6).contiguous()
    alpha = torch.empty(N * K + offset, device="cuda")[offset:].view(N, K)
    alpha.copy_(torch.randn(N, K, generator=gen, device="cuda") * 1.5)
    start = alpha.clone()
    grad, loss = fpq.fpq_round_learn_step(w, scale, fpq.E2M1, alpha, a, 1e-6, lr=lr)
    assert fpq.fpq_read_status() == fpq.OK
    wq, dwq = O.soft_weight(w.cpu().numpy(), scale.cpu().numpy(), O.E2M1, start.cpu().numpy())
    e = (torch.from_numpy(np.asarray(wq, dtype=np.float64)) - w.cpu().double()).cuda()
    d = torch.from_numpy(np.asarray(dwq, dtype=np.float64)).cuda()
    y = a.double() @ e.T
    assert float(loss[0]) == pytest.approx(float((y * y).mean()), rel=1e-5)
    data = 2.0 / (M * N) * (y.T @ a.double()) * d
    # what the regulariser adds, from a step on activations of zero
    reg, _ = fpq.fpq_round_learn_step(w, scale, fpq.E2M1, start.clone(), torch.zeros_like(a), 1e-6)
    assert float((grad.double() - reg.double() - data).norm()) <= 1e-5 * float(data.norm())
    if lr:
        assert torch.equal(alpha, start - lr * grad) or float((alpha - (start - lr * grad)).abs().max()) <= 1e-6 * float(alpha.abs().max())
    else:
        assert torch.equal(alpha, start)
