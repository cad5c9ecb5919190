"""The two forms of the encoding / bias search (Sec. V-A, Algorithm 1) around the size where the library changes
from applying every candidate to every element to sorting the elements, against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2408_06995_b200 as fpq

pytestmark = pytest.mark.gpu

# as in test_gpu_search.py: one FP32 rounding per error term at most, sums of 512 terms in FP32, then double; the
# sorted form works in double throughout
RTOL = 2e-6

FP8 = [fpq.Format(f.e, f.m, f.B, fpq.SAT_PAPER) for f in O.FP8_ENCODINGS]
FP4 = [fpq.Format(f.e, f.m, f.B, fpq.SAT_PAPER) for f in O.FP4_ENCODINGS]


def _search(x, encs, clips):
    mse, best = fpq.fpq_search_format(x, encs, torch.from_numpy(clips).cuda())
    return mse.cpu().numpy(), tuple(best.cpu().numpy())


def _data(kind, n, rng):
    x = rng.standard_normal(n).astype(np.float32)
    if kind == "wide":                     # many binades: most elements lie below the binned range
        x *= np.exp2(rng.uniform(-60, 0, n)).astype(np.float32)
    elif kind == "outlier":                # one entry far above the rest and above every clipping value
        x[n // 3] = 4e4
    elif kind == "zeros":                  # ReLU-like
        x[x < 0] = 0
    elif kind == "small":
        x *= np.float32(1e-18)
    return x


@pytest.mark.parametrize("kind", ["normal", "wide", "outlier", "zeros", "small"])
@pytest.mark.parametrize("n", [416666, 416667, 148 * 32768 + 5])
def test_both_forms_match_the_oracle(kind, n):
    x = _data(kind, n, np.random.default_rng(n))
    big = n > 1000000
    top = float(np.abs(x).max()) * (0.25 if kind == "outlier" else 1.0)
    clips = O.clip_candidates(top, 30)                     # 6 x 30: enough candidates for the sorted form
    pick = [0, 17, 29] if big else list(range(0, 30, 2))   # (the oracle checks some of them)
    got, best = _search(torch.from_numpy(x).cuda(), FP8 + FP4, clips)
    assert fpq.fpq_read_status() == fpq.OK
    want = O.search_mse(x, O.FP8_ENCODINGS + O.FP4_ENCODINGS, clips[pick])
    np.testing.assert_allclose(got[:, pick], want, rtol=RTOL, atol=0)
    assert best == O.select_encoding_and_bias(got)


def test_unaligned_tensor_and_repeatability():
    x = torch.from_numpy(_data("normal", 400002, np.random.default_rng(3))).cuda()[1:]
    clips = O.clip_candidates(float(x.abs().max()), 100)
    got, best = _search(x, FP8, clips)
    want = O.search_mse(x.cpu().numpy(), O.FP8_ENCODINGS, clips[::10])
    np.testing.assert_allclose(got[:, ::10], want, rtol=RTOL, atol=0)
    again, best2 = _search(x, FP8, clips)
    assert np.array_equal(got, again) and best == best2


def test_data_on_a_candidates_grid():
    # quantized data has (nearly) no error for its own format: nothing of the bins' width may be left
    f = O.FP8_ENCODINGS[2]
    rng = np.random.default_rng(4)
    clips = O.clip_candidates(8.3, 48)
    scale = np.float32(clips[47]) / np.float32(O.cmax(f))
    x = (rng.choice(O.decode_table(f), 400000).astype(np.float32) * scale).astype(np.float32)
    got, best = _search(torch.from_numpy(x).cuda(), FP8, clips)
    want = O.search_mse(x, O.FP8_ENCODINGS, clips)
    other = want > 1e-9
    np.testing.assert_allclose(got[other], want[other], rtol=RTOL, atol=0)
    # what is left of the matching candidate is FP32 rounding of scale * value: (2^-24 |x|)^2 per element
    assert got[2, 47] <= (2.0 ** -24 * 8.3) ** 2 and best == (2, 47)


def test_tensor_in_two_parts():
    # more than 2^24 elements
    n = (1 << 24) + 5
    x = torch.randn(n, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    x[-3] = 9.0
    clips = O.clip_candidates(float(x.abs().max()), 111)
    got, best = _search(x, FP4, clips)
    want = O.search_mse(x.cpu().numpy(), O.FP4_ENCODINGS, clips[[20, 60]])
    np.testing.assert_allclose(got[:, [20, 60]], want, rtol=RTOL, atol=0)
    assert best == O.select_encoding_and_bias(got)


def test_nan_in_a_large_tensor():
    x = torch.randn(200000, device="cuda")
    x[123456] = float("nan")
    got, best = _search(x, FP8, O.clip_candidates(4.0, 111))
    assert fpq.fpq_read_status() == fpq.ERR_NAN_INPUT
    assert np.isnan(got).all() and best == (-1, -1)


def _crowd(n, rng):
    # most elements in one bin, some of its neighbours with odd counts, thresholds of many candidates through it
    x = (1.0 + rng.integers(0, 4096, n) * 2.0 ** -23).astype(np.float32)
    x[:: 1000] = rng.uniform(0.25, 2.0, x[:: 1000].size)
    return x * rng.choice([-1.0, 1.0], n).astype(np.float32)


# 180 candidates: from 230445 elements on sorted, four shares up to 315000 and two up to 630000; a block sorts up to 61440
# elements at a time
@pytest.mark.parametrize("kind", ["normal", "crowd"])
@pytest.mark.parametrize("n", [230444, 230445, 315000, 315001, 630001, 148 * 61440, 148 * 61440 + 1])
def test_shares_and_pieces(kind, n):
    rng = np.random.default_rng(n)
    x = _data("normal", n, rng) if kind == "normal" else _crowd(n, rng)
    clips = O.clip_candidates(float(np.abs(x).max()), 30)
    pick = [3, 20] if n > 1000000 else [0, 7, 14, 21, 29]
    got, best = _search(torch.from_numpy(x).cuda(), FP8 + FP4, clips)
    assert fpq.fpq_read_status() == fpq.OK
    want = O.search_mse(x, O.FP8_ENCODINGS + O.FP4_ENCODINGS, clips[pick])
    np.testing.assert_allclose(got[:, pick], want, rtol=RTOL, atol=0)
    assert best == O.select_encoding_and_bias(got)
