"""Linear layers whose CTAs keep one column tile's weights and walk the row tiles: more tiles than CTAs, ragged last row
and column tiles, one to six chunks of the reduction, row lengths on both sides of the flat quantizer's rule."""
import numpy as np
import pytest

from paper_2408_06995_b200 import inputs as I
from _helpers import assert_close, gpu_layer, layer_scales, oracle_layer, sample_indices

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wfmt", ["e4m3", "e2m1"])
@pytest.mark.parametrize("M,K,N", [(9500, 64, 200), (9473, 320, 388), (6400, 104, 1156), (4800, 640, 640), (19000, 16, 132),
                                   (2500, 384, 2560)])
def test_against_the_oracle(M, K, N, wfmt):
    L = I.draw(I.linear_layer("columns", M, K, N, wfmt, rounding=(wfmt == "e2m1")), 31, 0, "normal", 0.02, True, 0.01, (0.001, 20.0))
    ws, xs = layer_scales(L)
    y = gpu_layer(L, ws, xs).reshape(-1)
    corners = np.concatenate([np.arange(2 * N), np.arange((M - 2) * N, M * N), np.arange(0, M * N, N)[::7] + N - 1])
    idx = sample_indices(y.size, 20000, 3, corners)
    yr, ab = oracle_layer(L, ws, xs, idx)
    assert_close(y[idx], yr, ab)
