"""Which form the rounding-learning step takes, without a GPU: A^T A needs room for its slices and for itself, so the size of
the workspace shows it."""
import pytest

import paper_2408_06995_b200 as fpq


def _with_gram(M, N, K):
    tiles = (K + 63) // 64
    size = fpq.fpq_round_learn_workspace_size(M, N, K)
    # the direct form's buffers: errors and derivatives, D and its transpose, A^T, and up to 64 slices of the gradient and of D
    return size, 8 * K * K + 8 * 4096 * tiles * (tiles + 1) // 2


# what measured faster (us, A^T A / direct: 43.8 / 59.6, 88.4 / 195.5, 22.9 / 38.0, 59.5 / 43.8, 68.5 / 50.8, 50.3 / 35.0, 132 / 72.8)
@pytest.mark.parametrize("M,N,K,gram", [(4096, 960, 320, True), (8192, 2560, 320, True), (1024, 512, 256, True), (8192, 320, 320, False),
                                        (2048, 640, 640, False), (94, 19, 1164, False), (1024, 2560, 640, False)])
def test_form(M, N, K, gram):
    size, least = _with_gram(M, N, K)
    odd = fpq.fpq_round_learn_workspace_size(M, N, K - 1)           # (rows of a multiple of 4 only)
    assert (size - odd >= least // 2) == gram
