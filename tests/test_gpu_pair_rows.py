"""Linear layers on CTA pairs (long reductions, weights of two terms): ragged rows, columns and reductions, rows of whole
and of partial chunks, every operand type, against the CPU oracle and against the general contraction."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2408_06995_b200 as fpq
from _helpers import assert_close

pytestmark = pytest.mark.gpu


def _o(f):
    return O.Format(f.exp_bits, f.man_bits, f.exp_bias, f.sat_mode)


@pytest.mark.parametrize("fx,fw,M,K,N", [
    (fpq.E4M3, fpq.E3M4, 2048, 2560, 640), (fpq.E4M3, fpq.E3M4, 300, 1152, 36), (fpq.E4M3, fpq.E2M5, 700, 500, 100),
    (fpq.E4M3, fpq.Format(5, 2, 16), 900, 386, 200), (fpq.E5M2, fpq.E3M4, 513, 700, 260), (fpq.E4M3, fpq.E2M1, 1300, 1540, 1000),
    (fpq.E4M3, fpq.E4M3, 2300, 900, 700), (fpq.E5M2, fpq.E5M2, 600, 1700, 1028), (fpq.E4M3, fpq.E1M2, 9217, 1300, 324),
    (fpq.E4M3, fpq.E4M3, 2300, 900, 1030), (fpq.E5M2, fpq.E5M2, 1200, 1700, 1028)])
def test_against_the_oracle_and_the_general_contraction(fx, fw, M, K, N):
    rng = np.random.default_rng(M + K + N)
    x = rng.standard_normal((M, K)).astype(np.float32)
    w = (rng.standard_normal((N, K)) * 0.02).astype(np.float32)
    bias = rng.standard_normal(N).astype(np.float32)
    ws = np.array([fpq.fpq_scale_from_max(float(v), fw) for v in np.abs(w).max(axis=1)], dtype=np.float32)
    xs = fpq.fpq_scale_from_max(float(np.abs(x).max()), fx)
    wd, wsd, xd, bd = [torch.from_numpy(v).cuda() for v in (w, ws, x, bias)]
    prep = fpq.fpq_prepare_weight(fpq.fpq_quantize_weight(wd, wsd, fw), fw, fpq.LINEAR, N, K)
    got = {}
    try:
        for policy in (fpq.PATH_TWO_KERNELS_NARROW, fpq.PATH_TWO_KERNELS, fpq.PATH_AUTO):
            fpq.fpq_set_path_policy(policy)
            got[policy] = fpq.fpq_linear(xd, prep, wsd, xs, fx, fw, bd, N).cpu().numpy()
    finally:
        fpq.fpq_set_path_policy(fpq.PATH_AUTO)
    assert fpq.fpq_read_status() == fpq.OK
    y = got[fpq.PATH_AUTO]
    assert np.array_equal(y, got[fpq.PATH_TWO_KERNELS])
    # exact products, FP32 sums in another order
    assert np.abs(y - got[fpq.PATH_TWO_KERNELS_NARROW]).max() <= 1e-5 * np.abs(y).max()
    rows = np.unique(np.concatenate([rng.integers(0, M, 20), [0, M - 1]]))
    idx = (rows[:, None] * N + np.arange(N)[None, :]).reshape(-1)
    yr, ab = O.linear(x, w, ws, xs, _o(fx), _o(fw), bias, None, idx)
    assert_close(y.reshape(-1)[idx], yr, ab)


# weights of two terms whose cheapest tile leaves no room for two stages of both terms' weights: the codes are still written
# once (the second half of the scratch stays as it was)
@pytest.mark.parametrize("fw,M,K,N", [(fpq.E3M4, 3000, 1280, 1280), (fpq.E3M4, 2300, 2561, 2560), (fpq.E2M5, 7000, 320, 2555)])
def test_two_terms_share_the_codes_with_wide_outputs(fw, M, K, N):
    gen = torch.Generator(device="cuda").manual_seed(N)
    x = torch.randn(M, K, generator=gen, device="cuda")
    w = torch.randn(N, K, generator=gen, device="cuda") * 0.02
    scale = (w.abs().amax(dim=1) / fpq.fpq_format_max(fw)).contiguous()
    prep = fpq.fpq_prepare_weight(fpq.fpq_quantize_weight(w, scale, fw), fw, fpq.LINEAR, N, K)
    bias = torch.randn(N, generator=gen, device="cuda")
    ws = torch.full((fpq.fpq_linear_workspace_size(M, N, K, fpq.E4M3, fw),), 0xAA, dtype=torch.uint8, device="cuda")
    got = fpq.fpq_linear(x, prep, scale, 0.01, fpq.E4M3, fw, bias, N, workspace=ws).clone()
    assert bool((ws[M * ((K + 15) // 16 * 16):] == 0xAA).all())
    try:
        fpq.fpq_set_path_policy(fpq.PATH_TWO_KERNELS_NARROW)
        want = fpq.fpq_linear(x, prep, scale, 0.01, fpq.E4M3, fw, bias, N, workspace=ws)
    finally:
        fpq.fpq_set_path_policy(fpq.PATH_AUTO)
    assert fpq.fpq_read_status() == fpq.OK
    # exact products, FP32 sums in another order
    assert float((got - want).abs().max()) <= 2e-5 * float(want.abs().max())
