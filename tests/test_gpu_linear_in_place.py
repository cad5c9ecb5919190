"""Linear layers whose output overlaps their input: what they give in a buffer of its own, whichever kernel that takes."""
import pytest
import torch

import paper_2408_06995_b200 as fpq

pytestmark = pytest.mark.gpu


# rows of every one-kernel form (1 to 8, 9 to 127) and of two kernels; `ahead`: floats between x and y, whole 16-byte pieces
@pytest.mark.parametrize("M,K,N,ahead", [(1, 1280, 1280, 0), (2, 1280, 1280, 0), (8, 320, 320, 0), (8, 640, 640, -640), (16, 320, 320, 0),
                                         (40, 1280, 1280, 0), (127, 640, 640, 0), (127, 640, 640, 4), (96, 320, 640, 320 * 95),
                                         (96, 640, 320, -320 * 95), (300, 640, 640, 0)])
@pytest.mark.parametrize("fw", [fpq.E4M3, fpq.E2M1])
@pytest.mark.parametrize("policy", [fpq.PATH_AUTO, fpq.PATH_FUSED])
def test_output_over_input(M, K, N, ahead, fw, policy):
    g = torch.Generator(device="cuda").manual_seed(M + K)
    x = torch.randn(M, K, generator=g, device="cuda")
    w = torch.randn(N, K, generator=g, device="cuda") * 0.02
    scale = (w.abs().amax(dim=1) / fpq.fpq_format_max(fw)).contiguous()
    prep = fpq.fpq_prepare_weight(fpq.fpq_quantize_weight(w, scale, fw), fw, fpq.LINEAR, N, K)
    try:
        fpq.fpq_set_path_policy(fpq.PATH_TWO_KERNELS)
        want = fpq.fpq_linear(x, prep, scale, 0.01, fpq.E4M3, fw, None, N)
        fpq.fpq_set_path_policy(policy)
        front = max(0, -ahead)
        room = torch.empty(front + max(M * K, ahead + M * N), device="cuda")
        inside, y = room[front:front + M * K].view(M, K), room[front + ahead:front + ahead + M * N].view(M, N)
        inside.copy_(x)
        fpq.fpq_linear(inside, prep, scale, 0.01, fpq.E4M3, fw, None, N, y)
    finally:
        fpq.fpq_set_path_policy(fpq.PATH_AUTO)
    assert fpq.fpq_read_status() == fpq.OK
    # the same exact products in FP32 sums of another order: fewer than K / 16 + 16 roundings, each of at most the sum of the
    # magnitudes, which a code has at most 1 / 16 (E4M3) or half of the largest step (E2M1: one scale) above its number
    terms = (1.07 * x.abs().double() + 1e-4) @ (1.07 * w.abs().double() + scale.double()[:, None]).T * 1.01
    assert bool(((y.double() - want.double()).abs() <= (K / 16 + 16) * 2.0 ** -24 * terms).all())
