"""Linear layers of a few rows, by default and on the routes without the kernel that takes most of them: one pass over the weights with
a column per warp or shared by two or four, ragged numbers of columns and of reduction steps, and the sizes beside the line
where the tensor cores take over; against the CPU oracle."""
import numpy as np
import pytest
import torch

import paper_2408_06995_b200 as fpq
from paper_2408_06995_b200 import inputs as I
from _helpers import assert_close, gpu_layer, layer_scales, oracle_layer, routes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N", [(1, 4, 1), (2, 260, 3), (3, 516, 7), (1, 1280, 641), (2, 1280, 1280), (4, 772, 639), (8, 5120, 66),
                                   (5, 2052, 33), (1, 4100, 2559), (2, 324, 2561), (8, 320, 1283), (8, 320, 2000), (3, 64, 9000),
                                   (1, 64, 9470), (6, 1284, 4100)])
@pytest.mark.parametrize("wfmt", ["e2m1", "e4m3"])
def test_few_rows(M, K, N, wfmt):
    L = I.draw(I.linear_layer("few", M, K, N, wfmt), 31, M, "silu", 0.02, True)
    ws, xs = layer_scales(L)
    yo, ab = oracle_layer(L, ws, xs)
    for route in routes(L):
        assert_close(gpu_layer(L, ws, xs, route=route), yo, ab)


def test_nan_in_a_row_is_reported():
    x = torch.randn(2, 1280, device="cuda")
    x[1, 1279] = float("nan")
    w = torch.randn(300, 1280, device="cuda")
    scale = (w.abs().amax(dim=1) / 6).contiguous()
    prep = fpq.fpq_prepare_weight(fpq.fpq_quantize_weight(w, scale, fpq.E2M1), fpq.E2M1, fpq.LINEAR, 300, 1280)
    y = fpq.fpq_linear(x, prep, scale, 0.01, fpq.E4M3, fpq.E2M1, None, 300)
    assert fpq.fpq_read_status() == fpq.ERR_NAN_INPUT
    assert fpq.fpq_read_status() == fpq.OK
    assert bool(torch.isfinite(y).all())


# tiles shared by clusters with several row tiles, ragged in rows, columns and chunks; few codes with 128-wide and 64-wide tiles
@pytest.mark.parametrize("M,K,N", [(200, 5120, 321), (513, 4990, 100), (129, 2560, 70), (16, 5100, 2600), (9, 2700, 3000), (25, 5120, 513),
                                   (64, 2304, 200)])
@pytest.mark.parametrize("wfmt", ["e2m1", "e4m3"])
def test_shared_tiles(M, K, N, wfmt):
    L = I.draw(I.linear_layer("shared", M, K, N, wfmt), 32, M, "silu", 0.02, True)
    ws, xs = layer_scales(L)
    yo, ab = oracle_layer(L, ws, xs)
    for route in routes(L):
        assert_close(gpu_layer(L, ws, xs, route=route), yo, ab)
