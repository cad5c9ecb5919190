"""Linear layers whose rows of output start anywhere (columns no multiple of 4): every remainder, ragged row tiles, one and
several tiles per CTA, weights resident and streamed, CTA pairs, weights of two terms; against the CPU oracle, outputs between guard bands."""
import pytest
import torch

import paper_2408_06995_b200 as fpq
from paper_2408_06995_b200 import inputs as I
from _helpers import assert_close, gpu_layer, layer_scales, oracle_layer, routes, sample_indices

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N", [(300, 64, 65), (33, 768, 130), (129, 320, 31), (1000, 128, 1027), (4100, 320, 637), (260, 2700, 333),
                                   (9000, 200, 66), (700, 383, 2570), (2500, 1536, 1283), (12, 640, 2),
                                   (3001, 1280, 1282), (2100, 2560, 639)])
@pytest.mark.parametrize("wfmt", ["e2m1", "e4m3"])
def test_ragged_columns(M, K, N, wfmt):
    L = I.draw(I.linear_layer("ragged", M, K, N, wfmt), 33, M, "silu", 0.02, True)
    ws, xs = layer_scales(L)
    idx = sample_indices(M * N, min(M * N, 200000), 7)
    yo, ab = oracle_layer(L, ws, xs, idx)
    for route in routes(L):
        assert_close(gpu_layer(L, ws, xs, route=route).reshape(-1)[idx], yo, ab)


@pytest.mark.parametrize("M,K,N", [(2048, 2560, 638), (300, 640, 65), (1111, 1300, 1283), (700, 640, 65)])
def test_two_terms(M, K, N):
    gen = torch.Generator(device="cuda").manual_seed(N)
    x = torch.randn(M, K, generator=gen, device="cuda")
    w = torch.randn(N, K, generator=gen, device="cuda") * 0.02
    scale = (w.abs().amax(dim=1) / fpq.fpq_format_max(fpq.E3M4)).contiguous()
    prep = fpq.fpq_prepare_weight(fpq.fpq_quantize_weight(w, scale, fpq.E3M4), fpq.E3M4, fpq.LINEAR, N, K)
    bias = torch.randn(N, generator=gen, device="cuda")
    got = fpq.fpq_linear(x, prep, scale, 0.01, fpq.E4M3, fpq.E3M4, bias, N).clone()
    try:
        fpq.fpq_set_path_policy(fpq.PATH_TWO_KERNELS_NARROW)
        want = fpq.fpq_linear(x, prep, scale, 0.01, fpq.E4M3, fpq.E3M4, bias, N)
    finally:
        fpq.fpq_set_path_policy(fpq.PATH_AUTO)
    assert fpq.fpq_read_status() == fpq.OK
    # the same products, FP32 sums of at most 5120 of them in another order: 5120 * 2^-24 of the sum of magnitudes at worst, a
    # hundredth of that in practice for terms of random sign
    assert float((got - want).abs().max()) <= 2e-5 * float(want.abs().max())


@pytest.mark.parametrize("M,K", [(37, 191), (37, 192), (5, 193), (129, 511), (40, 512), (9, 513), (3, 1025), (1, 4487), (600, 324)])
@pytest.mark.parametrize("fx", [fpq.E4M3, fpq.E5M2])
def test_row_codes(M, K, fx):
    # the standalone quantizer's codes, rows padded with zeros to a multiple of 16
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
