"""The row quantizer's codes for rows of every kind of length: whole 16-byte pieces, multiples of 4, others; one copy and two
(weights of two terms), both FP8 types, against the quantizer of single values."""
import pytest
import torch

import paper_2408_06995_b200 as fpq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K", [(1, 4), (3, 12), (700, 20), (37, 188), (37, 196), (5, 276), (1025, 340), (129, 516), (40, 1004), (2, 4100),
                                 (20001, 44), (37, 192), (9, 513), (600, 77)])
@pytest.mark.parametrize("fx", [fpq.E4M3, fpq.E5M2])
def test_row_codes(M, K, fx):
    x = torch.randn(M, K, device="cuda") * 3
    x[0, K - 1] = -0.0
    Kp = (K + 15) // 16 * 16
    ws = torch.full((M * Kp + 256,), 0xAA, dtype=torch.uint8, device="cuda")
    fpq.fpq_linear_quantize_input(x, 0.01, fx, fpq.E4M3, 64, ws)
    assert fpq.fpq_read_status() == fpq.OK
    want = torch.zeros(M, Kp, dtype=torch.uint8, device="cuda")
    want[:, :K] = fpq.fpq_quantize_act(x, 0.01, fx).view(torch.uint8).reshape(M, K)
    assert torch.equal(ws[:M * Kp].view(M, Kp), want)
    assert bool((ws[M * Kp:] == 0xAA).all())


@pytest.mark.parametrize("M,K", [(3, 4), (33, 132), (7, 384), (30, 1004), (65, 199)])
def test_codes_written_twice(M, K):
    # what a layer with weights of two terms leaves in its scratch, where it is too small for one copy
    x = torch.randn(M, K, device="cuda")
    w = torch.randn(64, K, device="cuda") * 0.02
    scale = (w.abs().amax(dim=1) / fpq.fpq_format_max(fpq.E3M4)).contiguous()
    prep = fpq.fpq_prepare_weight(fpq.fpq_quantize_weight(w, scale, fpq.E3M4), fpq.E3M4, fpq.LINEAR, 64, K)
    Kp = (K + 127) // 128 * 128
    ws = torch.full((fpq.fpq_linear_workspace_size(M, 64, K, fpq.E4M3, fpq.E3M4) + 256,), 0xAA, dtype=torch.uint8, device="cuda")
    fpq.fpq_linear(x, prep, scale, 0.01, fpq.E4M3, fpq.E3M4, None, 64, workspace=ws)
    assert fpq.fpq_read_status() == fpq.OK
    want = torch.zeros(M, 2, Kp, dtype=torch.uint8, device="cuda")
    want[:, :, :K] = fpq.fpq_quantize_act(x, 0.01, fpq.E4M3).view(torch.uint8).reshape(M, 1, K)
    assert torch.equal(ws[:M * 2 * Kp].view(M, 2, Kp), want)
    assert bool((ws[M * 2 * Kp:] == 0xAA).all())


def test_nan_is_code_zero_and_reported():
    x = torch.randn(50, 300, device="cuda")
    x[49, 299] = float("nan")
    ws = torch.full((50 * 304,), 0xAA, dtype=torch.uint8, device="cuda")
    fpq.fpq_linear_quantize_input(x, 0.01, fpq.E4M3, fpq.E4M3, 64, ws)
    assert fpq.fpq_read_status() == fpq.ERR_NAN_INPUT
    assert int(ws.view(50, 304)[49, 299]) == 0
