"""Convolutions on CTA pairs with column tiles of every width the library picks (32 .. 256 in steps of 32, a last tile of
less), one and two input tensors, one and two accumulators in tensor memory, and frames that are much of the image:
against the general contraction, whose products and order of additions are the same, bit for bit where it does not split
the reduction over a cluster, else within the rounding of the FP32 sums; and against the CPU oracle at one size."""
import numpy as np
import pytest
import torch

import paper_2408_06995_b200 as fpq
from paper_2408_06995_b200 import inputs as I
from _helpers import assert_close, gpu_layer, layer_scales, oracle_layer, sample_indices

pytestmark = pytest.mark.gpu


def _both(call):
    try:
        fpq.fpq_set_path_policy(fpq.PATH_TWO_KERNELS_NARROW)
        want = call().clone()
        fpq.fpq_set_path_policy(fpq.PATH_TWO_KERNELS)
        got = call().clone()
    finally:
        fpq.fpq_set_path_policy(fpq.PATH_AUTO)
    assert fpq.fpq_read_status() == fpq.OK
    # FP32 sums of at most 2^15 exact products in another order: 2^15 * 2^-24 of the sum of magnitudes at worst, a
    # hundredth of that in practice; outputs here are sums of K terms of random sign, so relative to the largest one
    assert float((got - want).abs().max()) <= 2e-5 * float(want.abs().max())


def _weights(gen, Co, K, fw):
    w = torch.randn(Co, K, generator=gen, device="cuda") * 0.05
    scale = (w.abs().amax(dim=1) / fpq.fpq_format_max(fw)).contiguous()
    return fpq.fpq_quantize_weight(w, scale, fw), scale


@pytest.mark.parametrize("B,C,H,W,Co", [(2, 320, 64, 64, 320), (2, 640, 32, 32, 640), (64, 192, 32, 32, 192), (8, 512, 32, 32, 512),
                                        (3, 320, 45, 45, 324), (5, 136, 30, 17, 100), (50, 416, 11, 11, 608), (2, 192, 7, 5, 288),
                                        (1, 256, 13, 96, 70), (16, 256, 32, 32, 256)])
@pytest.mark.parametrize("fw", [fpq.E4M3, fpq.E2M1])
def test_one_tensor(B, C, H, W, Co, fw):
    gen = torch.Generator(device="cuda").manual_seed(C + Co)
    x = torch.randn(B, C, H, W, generator=gen, device="cuda")
    codes, scale = _weights(gen, Co, C * 9, fw)
    prep = fpq.fpq_prepare_weight(codes, fw, fpq.CONV2D, Co, C, 3, 3)
    bias = torch.randn(Co, generator=gen, device="cuda")
    _both(lambda: fpq.fpq_conv2d(x, prep, scale, 0.01, fpq.E4M3, fw, bias, Co, 3, 3, 1, 1))


@pytest.mark.parametrize("B,C1,C2,res,Co,R", [(2, 640, 320, 64, 320, 3), (2, 640, 320, 32, 640, 3), (2, 1280, 640, 16, 1280, 3),
                                              (4, 100, 7, 33, 250, 3), (3, 128, 300, 9, 96, 3), (2, 320, 640, 64, 320, 1),
                                              (2, 320, 320, 64, 4, 3), (9, 130, 128, 20, 32, 3)])
def test_two_tensors(B, C1, C2, res, Co, R):
    fw = fpq.E2M1
    gen = torch.Generator(device="cuda").manual_seed(C1 + C2)
    x1 = torch.randn(B, C1, res, res, generator=gen, device="cuda")
    x2 = torch.randn(B, C2, res, res, generator=gen, device="cuda") * 3
    codes, scale = _weights(gen, Co, (C1 + C2) * R * R, fw)
    prep = fpq.fpq_prepare_weight_split(codes, fw, Co, C1, C2, R, R)
    bias = torch.randn(Co, generator=gen, device="cuda")
    y = torch.empty(B, Co, res, res, device="cuda")
    ws = torch.empty(fpq.fpq_conv2d_split_workspace_size(B, C1, C2, res, res, Co, R, R, R // 2, 1, fpq.E4M3, fw),
                     dtype=torch.uint8, device="cuda")
    _both(lambda: fpq.fpq_conv2d_split(x1, 0.01, x2, 0.03, prep, scale, fpq.E4M3, fw, bias, y, R, R, R // 2, 1, ws))


def test_small_frame_against_the_oracle():
    L = I.draw(I.conv_layer("frame", 9, 150, 7, 9, 104, 3, wfmt="e2m1", rounding=True), 21, 0, "silu", 0.03, True)
    ws, xs = layer_scales(L)
    y = gpu_layer(L, ws, xs).reshape(-1)
    idx = sample_indices(y.size, 20000, 5)
    yr, ab = oracle_layer(L, ws, xs, idx)
    assert_close(y[idx], np.asarray(yr), np.asarray(ab))


# few outputs: a tile of 32 columns, most of them past the last one or none
@pytest.mark.parametrize("B,C,H,W,Co,stride", [(2, 320, 64, 64, 4, 1), (16, 256, 32, 32, 32, 1), (28, 192, 10, 10, 1, 1), (28, 192, 10, 10, 31, 1),
                                               (8, 320, 64, 64, 32, 2), (8, 320, 64, 64, 3, 2)])
@pytest.mark.parametrize("fw", [fpq.E4M3, fpq.E2M1])
def test_few_outputs(B, C, H, W, Co, stride, fw):
    assert fpq.fpq_conv2d_contraction(B, C, H, W, Co, 3, 3, 1, stride, fpq.E4M3, fw) == fpq.CONTRACTION_PAIRS
    gen = torch.Generator(device="cuda").manual_seed(C + Co)
    x = torch.randn(B, C, H, W, generator=gen, device="cuda")
    codes, scale = _weights(gen, Co, C * 9, fw)
    prep = fpq.fpq_prepare_weight(codes, fw, fpq.CONV2D, Co, C, 3, 3)
    bias = torch.randn(Co, generator=gen, device="cuda")
    _both(lambda: fpq.fpq_conv2d(x, prep, scale, 0.01, fpq.E4M3, fw, bias, Co, 3, 3, 1, stride))


# stride 2: tiles of whole rows, parts of rows, several images; odd and even frames; one and several rounds
@pytest.mark.parametrize("B,C,H,W,Co", [(3, 320, 45, 77, 320), (2, 320, 64, 64, 320), (13, 128, 9, 8, 100), (1, 200, 7, 120, 256),
                                        (1, 64, 3, 253, 64), (1, 64, 3, 253, 72), (40, 96, 4, 3, 72), (9, 320, 31, 30, 640), (24, 192, 48, 48, 320)])
@pytest.mark.parametrize("fw,pad", [(fpq.E4M3, 1), (fpq.E2M1, 1), (fpq.E2M1, 0)])
def test_stride_two(B, C, H, W, Co, fw, pad):
    gen = torch.Generator(device="cuda").manual_seed(C + Co)
    x = torch.randn(B, C, H, W, generator=gen, device="cuda")
    codes, scale = _weights(gen, Co, C * 9, fw)
    prep = fpq.fpq_prepare_weight(codes, fw, fpq.CONV2D, Co, C, 3, 3)
    bias = torch.randn(Co, generator=gen, device="cuda")
    _both(lambda: fpq.fpq_conv2d(x, prep, scale, 0.01, fpq.E4M3, fw, bias, Co, 3, 3, pad, 2))


@pytest.mark.parametrize("B,C,H,W,Co", [(3, 130, 25, 41, 96), (7, 64, 11, 9, 40), (7, 64, 11, 9, 72)])
def test_stride_two_against_the_oracle(B, C, H, W, Co):
    L = I.draw(I.conv_layer("down", B, C, H, W, Co, 3, stride=2, wfmt="e2m1", rounding=True), 22, 0, "silu", 0.03, True)
    ws, xs = layer_scales(L)
    y = gpu_layer(L, ws, xs).reshape(-1)
    idx = sample_indices(y.size, 20000, 5)
    yr, ab = oracle_layer(L, ws, xs, idx)
    assert_close(y[idx], np.asarray(yr), np.asarray(ab))
