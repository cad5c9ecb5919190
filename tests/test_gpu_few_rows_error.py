"""Linear layers of few rows as one kernel are no further from 64-bit sums than the routes that such layers take without it."""
import numpy as np
import pytest
import torch

import paper_2408_06995_b200 as fpq

pytestmark = pytest.mark.gpu


TYPES = {"e4m3": (fpq.E4M3, torch.float8_e4m3fn, 448.0), "e5m2": (fpq.E5M2, torch.float8_e5m2, 57344.0)}


def _errors(M, K, fx, fw, seeds=6, N=1280):
    """2-norm errors, over several inputs, of the default route and of the one that never takes the kernel for few rows."""
    err = np.zeros(2)
    (gx, tx, cx), (gw, tw, cw) = TYPES[fx], TYPES[fw]
    for seed in range(seeds):
        g = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.nn.functional.silu(torch.randn(M, K, generator=g, device="cuda"))
        w = torch.randn(N, K, generator=g, device="cuda") * 0.02
        scale = (w.abs().amax(dim=1) / cw).contiguous()
        codes = fpq.fpq_quantize_weight(w, scale, gw)
        prep = fpq.fpq_prepare_weight(codes, gw, fpq.LINEAR, N, K)
        x_scale = float(np.float32(float(x.max()) / cx))
        q = (x * float(np.float32(1) / np.float32(x_scale))).clamp(-cx, cx).to(tx).double()
        want = q @ codes.view(tw).view(N, K).double().T * (scale.double() * x_scale)
        try:
            for i, policy in enumerate((fpq.PATH_AUTO, fpq.PATH_TWO_KERNELS)):
                fpq.fpq_set_path_policy(policy)
                y = fpq.fpq_linear(x, prep, scale, x_scale, gx, gw, None, N)
                err[i] += float((y.double() - want).norm() / want.norm()) / seeds
        finally:
            fpq.fpq_set_path_policy(fpq.PATH_AUTO)
    assert fpq.fpq_read_status() == fpq.OK
    return err


# E4M3 weights (with E2M1 ones the sums are exact up to the last rounding on either route): groups of 64 that a warp has alone or
# shares, sums of all eight warps, several groups per warp; rows of the CUDA-core form (up to 8) and of the two kernels
@pytest.mark.parametrize("K", [64, 96, 128, 132, 256, 260, 320, 640, 1280, 2560, 5120])
@pytest.mark.parametrize("M", [1, 2, 8, 40])
def test_error_against_64_bits(M, K):
    one, other = _errors(M, K, "e4m3", "e4m3")
    assert one <= other * (1 + 1e-9)
    assert one < 1.5e-7                                   # (a few roundings to FP32)


@pytest.mark.parametrize("M,K", [(2, 64), (40, 64), (8, 320), (40, 640), (2, 2560), (40, 2560)])
@pytest.mark.parametrize("fx,fw", [("e4m3", "e5m2"), ("e5m2", "e4m3"), ("e5m2", "e5m2")])
def test_error_with_e5m2(M, K, fx, fw):
    one, other = _errors(M, K, fx, fw)
    assert one <= other * (1 + 1e-9)
    assert one < 1.5e-7
