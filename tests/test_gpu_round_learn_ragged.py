"""The rounding-learning step at ragged sizes, with columns of very different size, and with operands that are not finite."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2408_06995_b200 as fpq

pytestmark = pytest.mark.gpu


def _inputs(M, N, K):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    w = torch.randn(N, K, generator=g, device="cuda") * 0.02
    a = torch.nn.functional.silu(torch.randn(M, K, generator=g, device="cuda") * 2)
    alpha = torch.randn(N, K, generator=g, device="cuda")
    return w, (w.abs().amax(dim=1) / 6).contiguous(), alpha, a


def _reference(w, scale, alpha, a):
    """Loss, gradient and what the rounding of the errors may add to it, in double."""
    wq, dwq = (torch.from_numpy(np.asarray(v, dtype=np.float64)).cuda() for v in
               O.soft_weight(w.cpu().numpy(), scale.cpu().numpy(), O.E2M1, alpha.cpu().numpy()))
    e, ad = wq - w.double(), a.double()
    d = ad @ e.T
    c = 2.0 / (a.shape[0] * w.shape[0]) * dwq
    noise = 2.0 ** -22 * (wq.abs() + w.double().abs())              # of an error: it is the difference of two FP32 numbers
    return (d * d).mean(), c * (d.T @ ad), c.abs() * (noise @ (ad.abs().T @ ad.abs()))


# a row and column; less and more than a tile of either product; few and many rows; rows of no multiple of 4 and of 16
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (31, 129, 47), (257, 127, 33), (600, 130, 129), (5000, 64, 95), (300, 513, 260),
                                   (8192, 130, 200), (9000, 257, 321), (2049, 300, 640), (40, 2000, 17)])
def test_sizes(M, N, K):
    w, scale, alpha, a = _inputs(M, N, K)
    grad, loss = fpq.fpq_round_learn_step(w, scale, fpq.E2M1, alpha, a, 0.0)
    assert fpq.fpq_read_status() == fpq.OK
    mse, want, noise = _reference(w, scale, alpha, a)
    assert float(loss[0]) == pytest.approx(float(mse), rel=1e-5)
    # the errors' own rounding, and that of the factors of the FP32 gradient
    assert bool(((grad.double() - want).abs() <= noise + 2.0 ** -19 * want.abs() + 1e-30).all())


def test_columns_of_very_different_size():
    w, scale, alpha, a = _inputs(700, 150, 132)
    a *= torch.exp2(torch.linspace(-60, 30, 132, device="cuda"))
    a[:, 7] = 0.0
    a[:, 8] = 1e-42
    grad, _ = fpq.fpq_round_learn_step(w, scale, fpq.E2M1, alpha, a, 0.0)
    _, want, noise = _reference(w, scale, alpha, a)
    assert bool(((grad.double() - want).abs() <= 2 * noise + 2.0 ** -19 * want.abs() + 1e-38).all())


@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_operands_that_are_not_finite(value):
    w, scale, alpha, a = _inputs(500, 140, 96)
    plain, _ = fpq.fpq_round_learn_step(w, scale, fpq.E2M1, alpha, a, 0.0)
    plain = plain.clone()
    bad = scale.clone()
    bad[131] = value                                     # an output channel whose scale is lost
    grad, loss = fpq.fpq_round_learn_step(w, bad, fpq.E2M1, alpha, a, 0.0)
    others = [n for n in range(140) if n != 131]
    assert torch.equal(grad[others], plain[others])
    fpq.fpq_read_status()
    # a calibration row with one such value: every gradient contains it
    a[77, 5] = value
    grad, loss = fpq.fpq_round_learn_step(w, scale, fpq.E2M1, alpha, a, 0.0)
    moves = torch.from_numpy(np.asarray(O.soft_weight(w.cpu().numpy(), scale.cpu().numpy(), O.E2M1, alpha.cpu().numpy())[1])).cuda() != 0
    assert not torch.isfinite(grad[moves]).any() and not bool(torch.isfinite(loss[0]))
    fpq.fpq_read_status()
