"""Convolutions either side of the lines between the one-kernel and the two-kernel route: each takes the route that the
measurements beside the rule give, and both routes agree."""
import pytest
import torch

import paper_2408_06995_b200 as fpq

pytestmark = pytest.mark.gpu
ONE, TWO = fpq.ROUTE_PAIR_FUSED, fpq.ROUTE_TWO_KERNELS


@pytest.mark.parametrize("B,C,H,W,Co,R,route", [
    (8, 128, 32, 32, 128, 3, TWO), (9, 128, 32, 32, 128, 3, ONE), (9, 128, 32, 32, 64, 3, TWO), (9, 64, 32, 32, 64, 3, ONE),
    (9, 128, 32, 32, 132, 3, TWO), (11, 128, 28, 28, 128, 3, TWO), (12, 64, 28, 28, 128, 3, ONE), (3, 65, 64, 64, 128, 3, TWO),
    (3, 64, 64, 64, 128, 3, ONE), (1, 100, 64, 64, 128, 1, ONE), (7, 100, 32, 32, 128, 1, TWO), (8, 100, 32, 32, 128, 1, ONE),
    (4, 128, 64, 64, 256, 1, ONE), (3, 128, 64, 64, 256, 1, TWO), (21, 128, 28, 28, 256, 1, ONE), (21, 128, 28, 28, 128, 1, TWO),
    (4, 129, 64, 64, 256, 1, TWO)])
def test_routes_agree(B, C, H, W, Co, R, route):
    assert fpq.fpq_conv2d_route(B, C, H, W, Co, R, R, R // 2, 1, fpq.E4M3, fpq.E2M1) == route
    gen = torch.Generator(device="cuda").manual_seed(C + Co)
    x = torch.randn(B, C, H, W, generator=gen, device="cuda")
    w = torch.randn(Co, C * R * R, generator=gen, device="cuda") * 0.05
    scale = (w.abs().amax(dim=1) / fpq.fpq_format_max(fpq.E2M1)).contiguous()
    prep = fpq.fpq_prepare_weight(fpq.fpq_quantize_weight(w, scale, fpq.E2M1), fpq.E2M1, fpq.CONV2D, Co, C, R, R)
    bias = torch.randn(Co, generator=gen, device="cuda")
    out = {}
    try:
        for policy in (fpq.PATH_AUTO, fpq.PATH_FUSED, fpq.PATH_TWO_KERNELS):
            fpq.fpq_set_path_policy(policy)
            out[policy] = fpq.fpq_conv2d(x, prep, scale, 0.01, fpq.E4M3, fpq.E2M1, bias, Co, R, R, R // 2, 1).clone()
    finally:
        fpq.fpq_set_path_policy(fpq.PATH_AUTO)
    assert fpq.fpq_read_status() == fpq.OK
    # the same products, FP32 sums of at most 1161 of them in another order: 1161 * 2^-24 of the sum of magnitudes at worst, a
    # hundredth of that in practice for terms of random sign
    want = out[fpq.PATH_TWO_KERNELS]
    for got in out.values():
        assert float((got - want).abs().max()) <= 2e-5 * float(want.abs().max())


# one tap: reductions shared by a cluster or not, on both sides of the rule
@pytest.mark.parametrize("B,C,H,W,Co,stride", [(8, 256, 20, 20, 300, 2), (15, 1344, 11, 40, 357, 2), (4, 1280, 8, 8, 640, 2),
                                               (2, 256, 16, 16, 256, 1), (2, 1280, 8, 8, 1280, 1)])
def test_one_tap_reductions(B, C, H, W, Co, stride):
    gen = torch.Generator(device="cuda").manual_seed(C + Co)
    x = torch.randn(B, C, H, W, generator=gen, device="cuda")
    w = torch.randn(Co, C, generator=gen, device="cuda") * 0.05
    scale = (w.abs().amax(dim=1) / fpq.fpq_format_max(fpq.E2M1)).contiguous()
    codes = fpq.fpq_quantize_weight(w, scale, fpq.E2M1)
    conv = fpq.fpq_prepare_weight(codes, fpq.E2M1, fpq.CONV2D, Co, C, 1, 1)
    got = fpq.fpq_conv2d(x, conv, scale, 0.01, fpq.E4M3, fpq.E2M1, None, Co, 1, 1, 0, stride)
    rows = x[:, :, ::stride, ::stride].permute(0, 2, 3, 1).reshape(-1, C).contiguous()
    lin = fpq.fpq_prepare_weight(codes, fpq.E2M1, fpq.LINEAR, Co, C)
    want = fpq.fpq_linear(rows, lin, scale, 0.01, fpq.E4M3, fpq.E2M1, None, Co)
    assert fpq.fpq_read_status() == fpq.OK
    got = got.permute(0, 2, 3, 1).reshape(-1, Co)
    # the same products, FP32 sums of at most 1344 of them in another order (as above)
    assert float((got - want).abs().max()) <= 2e-5 * float(want.abs().max())
