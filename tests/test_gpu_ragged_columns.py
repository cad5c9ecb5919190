"""Linear layers whose rows of output start anywhere (columns no multiple of 4): every remainder, ragged row tiles, one and
several tiles per CTA, weights resident and streamed; against the CPU oracle, outputs between guard bands."""
import pytest

from paper_2408_06995_b200 import inputs as I
from _helpers import assert_close, gpu_layer, layer_scales, oracle_layer, sample_indices

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N", [(300, 64, 65), (33, 768, 130), (129, 320, 31), (1000, 128, 1027), (4100, 320, 637), (260, 2700, 333),
                                   (9000, 200, 66), (700, 383, 2570), (2500, 1536, 1283), (12, 640, 2)])
@pytest.mark.parametrize("wfmt", ["e2m1", "e4m3"])
def test_ragged_columns(M, K, N, wfmt):
    L = I.draw(I.linear_layer("ragged", M, K, N, wfmt), 33, M, "silu", 0.02, True)
    ws, xs = layer_scales(L)
    y = gpu_layer(L, ws, xs).reshape(-1)
    idx = sample_indices(y.size, min(y.size, 200000), 7)
    yo, ab = oracle_layer(L, ws, xs, idx)
    assert_close(y[idx], yo, ab)
