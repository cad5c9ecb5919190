"""The rounding-learning step from A^T A against 64-bit sums of the very FP32 errors that it works with, on correlated
calibration rows with errors that cancel along them: its sums are as good as sums in double are."""
import numpy as np
import pytest
import torch

import paper_2408_06995_b200 as fpq

pytestmark = pytest.mark.gpu


def _case(kind, M, N, K, left, seed):
    """alpha = 0 has sigma = 1/2 and its derivative 1/4 without rounding, so that Wq is in the middle of a step of 2 (E2M1, from
    4 to 6) and the errors, one rounding each, are known here."""
    rng = np.random.default_rng(seed)
    noise = rng.standard_normal((M, K))
    low = rng.standard_normal((M, 32)) @ rng.standard_normal((32, K))
    a = {"rank": low, "noisy rank": low + 1e-3 * noise, "mean 500": noise + 500.0}[kind].astype(np.float32)
    scale = (0.01 * rng.uniform(0.5, 1.0, N)).astype(np.float32)
    e = rng.standard_normal((N, K)) * 0.06
    _, s, vt = np.linalg.svd(a.astype(np.float64), full_matrices=False)
    lead = vt[s > 1e-2 * s[0]]
    e -= (1 - left) * (e @ lead.T) @ lead
    g = scale.astype(np.float64)[:, None]
    w = (g * (np.where(rng.random((N, K)) < 0.5, 5.0, -5.0) - np.clip(e, -0.9, 0.9))).astype(np.float32)
    wq = g * (np.where(w > 0, 5.0, -5.0))
    return w, scale, a, (wq - w).astype(np.float32), 0.5 * g


@pytest.mark.parametrize("kind", ["rank", "noisy rank", "mean 500"])
@pytest.mark.parametrize("left", [1.0, 1e-3, 0.0])
@pytest.mark.parametrize("M,N,K", [(1024, 512, 256), (1100, 700, 324), (4096, 960, 320)])
def test_sums_in_double(kind, left, M, N, K):
    w, scale, a, e, dwq = _case(kind, M, N, K, left, M + K)
    alpha = torch.zeros(N, K, device="cuda")
    grad, loss = fpq.fpq_round_learn_step(*(torch.from_numpy(v).cuda() for v in (w, scale)), fpq.E2M1, alpha, torch.from_numpy(a).cuda(), 0.0)
    assert fpq.fpq_read_status() == fpq.OK
    a64, e64 = a.astype(np.float64), e.astype(np.float64)
    d = a64 @ e64.T
    # A sum of n terms in double: some sqrt(n) roundings of random sign, each 2^-53 of the terms' magnitudes.  Those of an entry of
    # A^T A are the same for all rows of E; six standard deviations, and the roundings of the loss itself.
    u = 2.0 ** -53
    s_abs = np.abs(a64).T @ np.abs(a64)
    through = u * np.sqrt(M) * np.linalg.norm((e64.T @ e64) * s_abs)
    product = u * np.sqrt(K) * (np.abs(e64) @ s_abs)                  # of an entry of E (A^T A)
    bound = 6 * (through + np.linalg.norm(product * e64)) / (M * N)
    mse = float(loss[0])
    assert abs(mse - np.mean(d * d)) <= bound + 1e-12 * mse
    # the gradient: as above, and three roundings to FP32
    want = 2.0 / (M * N) * (d.T @ a64) * dwq
    entry = u * np.sqrt(M) * np.sqrt((e64 ** 2) @ (s_abs ** 2)) + product
    err = np.linalg.norm(grad.cpu().numpy() - want)
    assert err <= np.linalg.norm(2.0 / (M * N) * 6 * entry * dwq) + 3 * 2.0 ** -24 * np.linalg.norm(want)


@pytest.mark.parametrize("M,N,K", [(600, 40, 47), (600, 40, 48), (3000, 300, 321)])
def test_scales_whose_reciprocal_overflows(M, N, K):
    g = torch.Generator(device="cuda").manual_seed(K)
    w, a = torch.randn(N, K, generator=g, device="cuda") + 3.0, torch.randn(M, K, generator=g, device="cuda")
    w[w == 0] = 1.0
    scale = torch.full((N,), 1.0, device="cuda")
    scale[N // 2] = 1e-41                                # weight / scale is infinite and is clipped; nothing is not a number
    fpq.fpq_round_learn_step(w, scale, fpq.E2M1, torch.zeros(N, K, device="cuda"), a, 0.0)
    assert fpq.fpq_read_status() == fpq.OK
