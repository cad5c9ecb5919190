"""Layers whose launches overlap the end of the kernel in front of them: every layer reads what the one before it wrote
(activations, the shared workspace, weights prepared or copied just before), so results must equal those of the same
calls with the GPU idle in between, bit for bit."""
import pytest
import torch

import paper_2408_06995_b200 as fpq

pytestmark = pytest.mark.gpu


def _weights(gen, N, K, fw, conv=None):
    w = torch.randn(N, K, generator=gen, device="cuda") * 0.05
    scale = (w.abs().amax(dim=1) / fpq.fpq_format_max(fw)).contiguous()
    codes = fpq.fpq_quantize_weight(w, scale, fw)
    if conv:
        return fpq.fpq_prepare_weight(codes, fw, fpq.CONV2D, N, K // 9, 3, 3), scale
    return fpq.fpq_prepare_weight(codes, fw, fpq.LINEAR, N, K), scale


def _linear_chain(wait, fw, M, widths, spare):
    gen = torch.Generator(device="cuda").manual_seed(7)
    x = torch.randn(M, widths[0], generator=gen, device="cuda")
    ws = torch.empty(1 << 24, dtype=torch.uint8, device="cuda")
    for K, N in zip(widths, widths[1:]):
        w, scale = _weights(gen, N, K, fw)
        spare[: w.numel()].copy_(w)                       # the layer reads weights that a copy has only just written
        wait()
        x = fpq.fpq_linear(x, spare, scale, 0.02, fpq.E4M3, fw, None, N, None, ws)
        spare.fill_(0)                                    # ... and that are overwritten right behind it
        wait()
    return x


def _conv_chain(wait, fw, B, res, widths, spare):
    gen = torch.Generator(device="cuda").manual_seed(8)
    x = torch.randn(B, widths[0], res, res, generator=gen, device="cuda")
    ws = torch.empty(1 << 25, dtype=torch.uint8, device="cuda")
    for C, Co in zip(widths, widths[1:]):
        w, scale = _weights(gen, Co, C * 9, fw, conv=True)
        spare[: w.numel()].copy_(w)
        wait()
        x = fpq.fpq_conv2d(x, spare, scale, 0.02, fpq.E4M3, fw, None, Co, 3, 3, 1, 1, None, ws)
        spare.fill_(0)
        wait()
    return x


@pytest.mark.parametrize("fw", [fpq.E4M3, fpq.E2M1, fpq.E3M4])
@pytest.mark.parametrize("M", [2, 33, 2048])
def test_chain_of_linear_layers(M, fw):
    widths = [320, 960, 128, 1280, 64, 2560, 320]
    spare = torch.empty(1 << 23, dtype=torch.uint8, device="cuda")
    want = _linear_chain(torch.cuda.synchronize, fw, M, widths, spare)
    for _ in range(3):
        assert torch.equal(_linear_chain(lambda: None, fw, M, widths, spare), want)
    assert fpq.fpq_read_status() == fpq.OK


@pytest.mark.parametrize("fw", [fpq.E4M3, fpq.E2M1])
@pytest.mark.parametrize("B,res", [(16, 32), (2, 8), (3, 19)])
def test_chain_of_convolutions(B, res, fw):
    widths = [128, 128, 256, 256, 64, 320]
    spare = torch.empty(1 << 23, dtype=torch.uint8, device="cuda")
    want = _conv_chain(torch.cuda.synchronize, fw, B, res, widths, spare)
    for _ in range(3):
        assert torch.equal(_conv_chain(lambda: None, fw, B, res, widths, spare), want)
    assert fpq.fpq_read_status() == fpq.OK
