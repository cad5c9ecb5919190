"""Linear layers of few rows as one kernel: at the edges of its blocks (8 and 16 rows, 16, 32 and 64 columns, 64 and 512 elements of
the reduction), for all operand types, against exact sums of the same codes and against the two-kernel route."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2408_06995_b200 as fpq

pytestmark = pytest.mark.gpu

FORMATS = {"e4m3": (fpq.E4M3, O.E4M3), "e5m2": (fpq.E5M2, O.E5M2), "e2m1": (fpq.E2M1, O.E2M1), "e1m2": (fpq.E1M2, O.E1M2)}


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


def _run(x, w, ws, xs, b, fx, fw, policy):
    M, K = x.shape
    N = w.shape[0]
    gfx, gfw = FORMATS[fx][0], FORMATS[fw][0]
    sc = torch.from_numpy(ws).cuda()
    prep = fpq.fpq_prepare_weight(fpq.fpq_quantize_weight(torch.from_numpy(w).cuda(), sc, gfw), gfw, fpq.LINEAR, N, K)
    y = torch.full((M + 2, N), float("nan"), device="cuda")
    ws_ = torch.empty(max(256, fpq.fpq_linear_workspace_size(M, N, K, gfx, gfw)), dtype=torch.uint8, device="cuda")
    try:
        fpq.fpq_set_path_policy(policy)
        fpq.fpq_linear(torch.from_numpy(x).cuda(), prep, sc, xs, gfx, gfw, None if b is None else torch.from_numpy(b).cuda(), N, y[:M], ws_)
    finally:
        fpq.fpq_set_path_policy(fpq.PATH_AUTO)
    assert bool(torch.isnan(y[M:]).all())                # nothing behind the output
    return y[:M].cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("M,K,N", [(1, 4, 1), (7, 60, 15), (8, 64, 16), (9, 68, 17), (16, 512, 33), (17, 516, 64), (33, 1028, 65), (64, 320, 129),
                                   (100, 576, 96), (127, 96, 160), (3, 2052, 31), (2, 1280, 1280), (126, 8, 40)])
@pytest.mark.parametrize("fx,fw", [("e4m3", "e4m3"), ("e4m3", "e2m1"), ("e4m3", "e5m2"), ("e5m2", "e4m3"), ("e5m2", "e2m1"), ("e5m2", "e5m2"),
                                   ("e4m3", "e1m2")])
def test_matches_sums_of_the_codes(M, K, N, fx, fw):
    x, w, ws, xs, b = _layer(M, K, N, fw, M + K + N, fx, bias=(M + K) % 3 != 0)
    y = _run(x, w, ws, xs, b, fx, fw, fpq.PATH_AUTO)
    two = _run(x, w, ws, xs, b, fx, fw, fpq.PATH_TWO_KERNELS)
    assert fpq.fpq_read_status() == fpq.OK
    # both are FP32 sums of the same K exact products: K roundings of at most the sum of their magnitudes each, and two ulps
    # for scale and bias; that sum is at most max |q(x)| max |w| K times the scales
    terms = np.abs(x).max(axis=1, keepdims=True).astype(np.float64) * np.abs(w).max(axis=1)[None].astype(np.float64) * K * 1.07
    tol = (K / 16 + 16) * 2.0 ** -24 * terms + 2 * np.spacing(np.abs(two).astype(np.float32))
    assert np.all(np.abs(y - two) <= tol)


def test_not_a_number_counts_as_zero_and_is_reported():
    x, w, ws, xs, b = _layer(20, 200, 48, "e4m3", 5)
    clean = x.copy()
    clean[3, 17] = clean[19, 199] = 0.0
    want = _run(clean, w, ws, xs, b, "e4m3", "e4m3", fpq.PATH_AUTO)
    assert fpq.fpq_read_status() == fpq.OK
    x[3, 17] = x[19, 199] = np.nan
    got = _run(x, w, ws, xs, b, "e4m3", "e4m3", fpq.PATH_AUTO)
    assert fpq.fpq_read_status() == fpq.ERR_NAN_INPUT
    assert np.array_equal(got, want)
    x[3, 17], x[19, 199] = np.inf, -np.inf               # saturate
    clean[3, 17], clean[19, 199] = 448 * xs * 2, -448 * xs * 2
    assert np.array_equal(_run(x, w, ws, xs, b, "e4m3", "e4m3", fpq.PATH_AUTO), _run(clean, w, ws, xs, b, "e4m3", "e4m3", fpq.PATH_AUTO))
    assert fpq.fpq_read_status() == fpq.OK
