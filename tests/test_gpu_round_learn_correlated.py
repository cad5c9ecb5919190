"""The loss of the rounding-learning step on correlated calibration rows (few distinct rows, low rank, a large common
mean) and weight errors that cancel along them, which is where descent leads: never negative, and as accurate as the sum of
the squared output errors."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2408_06995_b200 as fpq

pytestmark = pytest.mark.gpu


def _rows(kind, M, K, rng):
    noise = rng.standard_normal((M, K))
    if kind == "repeated":
        return rng.standard_normal((4, K))[rng.integers(0, 4, M)]
    if kind == "rank":
        return rng.standard_normal((M, 32)) @ rng.standard_normal((32, K))
    if kind == "noisy rank":
        return rng.standard_normal((M, 32)) @ rng.standard_normal((32, K)) + 1e-3 * noise
    return noise + {"mean 10": 10.0, "mean 50": 50.0, "mean 500": 500.0}[kind]


def _case(kind, M, N, K, left, seed):
    """Weights in the middle of their step and decisions whose errors keep only `left` of their part along the rows' leading
    directions."""
    rng = np.random.default_rng(seed)
    a = _rows(kind, M, K, rng).astype(np.float32)
    f = rng.uniform(0.3, 0.7, (N, K))
    scale = (0.01 * rng.uniform(0.5, 1.0, N)).astype(np.float32)
    w = (np.where(rng.random((N, K)) < 0.5, 4 + 2 * f, -6 + 2 * f) * scale[:, None]).astype(np.float32)
    e = rng.standard_normal((N, K)) * 0.06
    _, s, vt = np.linalg.svd(a.astype(np.float64), full_matrices=False)
    lead = vt[s > 1e-2 * s[0]][: K // 2]
    h = np.clip(f + e - (1 - left) * (e @ lead.T) @ lead, 0.02, 0.98)
    return w, scale, np.log(h / (1 - h)).astype(np.float32), a


@pytest.mark.parametrize("kind", ["repeated", "rank", "noisy rank", "mean 10", "mean 50", "mean 500"])
@pytest.mark.parametrize("left", [1.0, 0.1, 1e-3, 0.0])
@pytest.mark.parametrize("M,N,K", [(1024, 200, 160), (1100, 700, 324)])
def test_loss_is_that_of_the_squared_errors(kind, left, M, N, K):
    w, scale, alpha, a = _case(kind, M, N, K, left, K)
    d = [torch.from_numpy(v).cuda() for v in (w, scale, alpha, a)]
    grad, loss = fpq.fpq_round_learn_step(d[0], d[1], fpq.E2M1, d[2], d[3], 0.0)
    assert fpq.fpq_read_status() == fpq.OK
    r = O.round_learn_step(w, scale, O.E2M1, alpha, a, 0.0)
    mse = float(loss[0])
    assert mse >= 0.0
    # An error is a difference of two FP32 numbers (the soft weight, some four roundings, and the weight): 2^-22 of their
    # magnitudes at worst, of random sign, so that those of a row's K terms add up like their squares.  An output error is a
    # sum of K products, here at FP32 accuracy: 4e-6 of the value it has, as for rows without correlation.
    a64, w64 = a.astype(np.float64), w.astype(np.float64)
    noise = 2.0 ** -22 * np.sqrt(np.mean((a64 ** 2) @ ((np.abs(w64) + np.abs(r["wq"])) ** 2).T))
    assert abs(np.sqrt(mse) - np.sqrt(r["mse"])) <= noise + 4e-6 * np.sqrt(r["mse"])
    # the gradient's two contractions: the same noise of the errors, through D^T A
    dwq = np.abs(O.soft_weight(w, scale, O.E2M1, alpha)[1])
    through = 2.0 / (M * N) * M * K * noise * np.sqrt(np.mean(a64 ** 2)) * np.sqrt(np.mean(dwq ** 2))
    err = np.linalg.norm(grad.cpu().numpy().astype(np.float64) - r["grad"]) / np.sqrt(N * K)
    assert err <= through + 1e-5 * np.linalg.norm(r["grad"]) / np.sqrt(N * K)
