"""Linear layers of few rows as one kernel: blocks of 8 and 16 rows by 16, 32 and 64 columns with ragged rows, columns and
reductions, sums of a group of 64 in one warp and in four, for all operand types, against 64-bit sums of the same codes."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2408_06995_b200 as fpq

pytestmark = pytest.mark.gpu

FORMATS = {"e4m3": (fpq.E4M3, O.E4M3), "e5m2": (fpq.E5M2, O.E5M2), "e2m1": (fpq.E2M1, O.E2M1), "e1m2": (fpq.E1M2, O.E1M2)}
PAIRS = [("e4m3", "e4m3"), ("e4m3", "e2m1"), ("e4m3", "e5m2"), ("e5m2", "e4m3"), ("e5m2", "e2m1"), ("e5m2", "e5m2"), ("e4m3", "e1m2")]


def _layer(M, K, N, fw, seed, fx="e4m3", bias=True):
    rng = np.random.default_rng(seed)
    x = (rng.standard_normal((M, K)) * 2).astype(np.float32)
    x[rng.random((M, K)) < 0.05] = -1e-9                 # rounds to minus zero
    w = (rng.standard_normal((N, K)) * 0.02).astype(np.float32)
    gfw, ofw = FORMATS[fw]
    ws = np.array([O.scale_from_max(v, ofw) for v in np.abs(w).max(axis=1) + 1e-12], dtype=np.float32)
    xs = float(O.scale_from_max(float(np.abs(x).max()), FORMATS[fx][1]))
    b = (rng.standard_normal(N) * 0.1).astype(np.float32) if bias else None
    return x, w, ws, xs, b


def _run(x, w, ws, xs, b, fx, fw, policy=fpq.PATH_AUTO, out_scale=None):
    M, K = x.shape
    N = w.shape[0]
    gfx, gfw = FORMATS[fx][0], FORMATS[fw][0]
    sc = torch.from_numpy(ws).cuda()
    prep = fpq.fpq_prepare_weight(fpq.fpq_quantize_weight(torch.from_numpy(w).cuda(), sc, gfw), gfw, fpq.LINEAR, N, K)
    if out_scale is not None:
        sc = torch.from_numpy(out_scale).cuda()
    y = torch.full((M + 2, N), float("nan"), device="cuda")
    ws_ = torch.empty(max(256, fpq.fpq_linear_workspace_size(M, N, K, gfx, gfw)), dtype=torch.uint8, device="cuda")
    try:
        fpq.fpq_set_path_policy(policy)
        fpq.fpq_linear(torch.from_numpy(x).cuda(), prep, sc, xs, gfx, gfw, None if b is None else torch.from_numpy(b).cuda(), N, y[:M], ws_)
    finally:
        fpq.fpq_set_path_policy(fpq.PATH_AUTO)
    assert bool(torch.isnan(y[M:]).all())                # nothing behind the output
    return y[:M].cpu().numpy().astype(np.float64)


def _sums(x, w, ws, xs, b, fx, fw):
    """The layer in double from the oracle's codes, and the sums of the magnitudes of the terms."""
    (M, K), N = x.shape, w.shape[0]
    ofx, ofw = FORMATS[fx][1], FORMATS[fw][1]
    xc = O.quantize_act(x.reshape(-1), xs, ofx)
    wc = O.quantize_weight(w, ws, ofw)
    if ofw.bits == 4:
        wc = np.stack([wc & 15, wc >> 4], axis=-1)
    xv = torch.from_numpy(O.decode_table(ofx)[xc.reshape(M, -1)[:, :K]]).double().cuda()
    wv = torch.from_numpy(O.decode_table(ofw)[wc.reshape(N, -1)[:, :K]]).double().cuda()
    scale = torch.from_numpy(ws).double().cuda() * float(np.float32(xs))
    y, terms = (xv @ wv.T) * scale, (xv.abs() @ wv.abs().T) * scale
    if b is not None:
        y = y + torch.from_numpy(b).double().cuda()
    return y.cpu().numpy(), terms.cpu().numpy()


# by blocks (rows x columns); up to 64 elements, or 143 with up to 8 rows, a group of 64 is summed in four warps
SHAPES = [
    (7, 60, 15), (76, 44, 79), (5, 140, 47), (8, 132, 33),                                # 8 x 16, short
    (9, 68, 17), (16, 512, 33), (17, 516, 64), (33, 1028, 65), (20, 1900, 351), (127, 96, 160), (2, 1280, 1280),       # 8 x 16
    (8, 8, 3059), (113, 52, 253),                                                         # 8 x 32, short
    (75, 540, 268), (116, 4688, 191),                                                     # 8 x 32
    (6, 72, 6918), (8, 176, 7296), (36, 2788, 1726),                                      # 8 x 64, the first short
    (125, 24, 1679), (33, 60, 1432), (50, 440, 3156), (97, 192, 1993),                    # 16 x 32, the first two short
    (33, 1392, 2946), (109, 1644, 677)]                                                   # 16 x 64


@pytest.mark.parametrize("M,K,N", SHAPES)
@pytest.mark.parametrize("fx,fw", PAIRS)
def test_matches_sums_of_the_codes(M, K, N, fx, fw):
    x, w, ws, xs, b = _layer(M, K, N, fw, M + K + N, fx, bias=(M + K) % 3 != 0)
    want, terms = _sums(x, w, ws, xs, b, fx, fw)
    form = fpq.fpq_linear_contraction(M, N, K, FORMATS[fx][0], FORMATS[fw][0])
    assert form == fpq.CONTRACTION_FEW_ROWS or (M <= 8 and form == fpq.CONTRACTION_CUDA_CORES)
    y = _run(x, w, ws, xs, b, fx, fw)
    assert fpq.fpq_read_status() == fpq.OK
    # On its way a product is part of four sums of an MMA (cut off: 2^-23 of the magnitudes each), one addition per 512 elements and
    # three of the warps' sums (2^-24 each); then come the scales' product, theirs with the sum, and the bias.
    n = 4 + (K / 512 + 1 + 3) / 2
    assert np.all(np.abs(y - want) <= n * 2.0 ** -23 * terms + 2 * np.spacing(np.abs(want).astype(np.float32)) + 2.0 ** -23 * np.abs(want))
    if form == fpq.CONTRACTION_FEW_ROWS:
        # the routes without this kernel, with at most K / 32 + 5 roundings of their own
        two = _run(x, w, ws, xs, b, fx, fw, fpq.PATH_TWO_KERNELS)
        assert np.all(np.abs(y - two) <= (n + K / 32 + 5) * 2.0 ** -23 * terms + 2 * np.spacing(np.abs(two).astype(np.float32)))


@pytest.mark.parametrize("M,K,N", [(1, 4, 1), (100, 576, 96), (3, 2052, 31), (126, 8, 40), (64, 320, 129)])
@pytest.mark.parametrize("fx,fw", PAIRS)
def test_smallest_and_plain_sizes(M, K, N, fx, fw):
    x, w, ws, xs, b = _layer(M, K, N, fw, M + K + N, fx)
    want, terms = _sums(x, w, ws, xs, b, fx, fw)
    y = _run(x, w, ws, xs, b, fx, fw)
    assert fpq.fpq_read_status() == fpq.OK
    # (either of the kernels for few rows: at most K / 32 + 5 FP32 roundings on the CUDA cores, see above for the other)
    n = max(4 + (K / 512 + 4) / 2, (K / 32 + 5) / 2)
    assert np.all(np.abs(y - want) <= n * 2.0 ** -23 * terms + 2 * np.spacing(np.abs(want).astype(np.float32)) + 2.0 ** -23 * np.abs(want))


@pytest.mark.parametrize("M,K,N", [(9, 1280, 40), (20, 1900, 351), (33, 60, 1432), (33, 1392, 2946)])
@pytest.mark.parametrize("fx,fw", [("e4m3", "e4m3"), ("e5m2", "e5m2")])
def test_scales_that_overflow(M, K, N, fx, fw):
    x, w, ws, xs, b = _layer(M, K, N, fw, 6, fx)
    out = ws.copy()
    out[[0, 7, 11, 14, N - 1]] = [np.inf, 3e38, -np.inf, 3e38 / 64, np.nan]
    x, xs = x * np.float32(1024), xs * 1024              # (the product of the scales overflows, or the result does)
    assert fpq.fpq_linear_contraction(M, N, K, FORMATS[fx][0], FORMATS[fw][0]) == fpq.CONTRACTION_FEW_ROWS
    y, two = (_run(x, w, ws, xs, b, fx, fw, policy, out) for policy in (fpq.PATH_AUTO, fpq.PATH_TWO_KERNELS))
    assert np.isinf(y).any()
    for n in (0, 7, 11, 14, N - 1):
        assert np.array_equal(np.where(np.isfinite(y[:, n]), 0.0, y[:, n]), np.where(np.isfinite(two[:, n]), 0.0, two[:, n]), equal_nan=True)
    fpq.fpq_read_status()


# a NaN in either group of eight rows of a block, in the last row and the last column, in sums of one warp and of four
@pytest.mark.parametrize("M,K,N", [(20, 200, 48), (109, 1644, 677), (97, 192, 1993), (33, 60, 1432), (8, 132, 33), (75, 540, 268)])
@pytest.mark.parametrize("fx,fw", PAIRS)
def test_not_a_number_counts_as_zero_and_is_reported(M, K, N, fx, fw):
    x, w, ws, xs, b = _layer(M, K, N, fw, 5, fx)
    rows = [3, min(12, M - 2), M - 1]
    cols = [K // 3, K // 2 + 1, K - 1]
    clean = x.copy()
    clean[rows, cols] = 0.0
    want = _run(clean, w, ws, xs, b, fx, fw)
    assert fpq.fpq_read_status() == fpq.OK
    x[rows, cols] = np.nan
    got = _run(x, w, ws, xs, b, fx, fw)
    assert fpq.fpq_read_status() == fpq.ERR_NAN_INPUT
    assert np.array_equal(got, want)
    most = float(O.cmax(FORMATS[fx][1]))
    x[rows, cols] = [np.inf, -np.inf, np.inf]            # saturate
    clean[rows, cols] = [most * xs * 2, -most * xs * 2, most * xs * 2]
    assert np.array_equal(_run(x, w, ws, xs, b, fx, fw), _run(clean, w, ws, xs, b, fx, fw))
    assert fpq.fpq_read_status() == fpq.OK
