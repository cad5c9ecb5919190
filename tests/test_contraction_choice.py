"""Which contraction the library picks, without a GPU: the shapes that the GPU tests of one kernel rely on take that kernel,
or those tests would compare another one with itself."""
import pytest

import paper_2408_06995_b200 as fpq

E4M3, E5M2, E2M1, E3M4, E2M5, E1M2 = fpq.E4M3, fpq.E5M2, fpq.E2M1, fpq.E3M4, fpq.E2M5, fpq.E1M2
GENERAL, PAIRS, CUDA_CORES, OTHER, FEW_ROWS = (fpq.CONTRACTION_GENERAL, fpq.CONTRACTION_PAIRS, fpq.CONTRACTION_CUDA_CORES,
                                               fpq.CONTRACTION_OTHER, fpq.CONTRACTION_FEW_ROWS)


# test_gpu_pair_rows.py and test_gpu_ragged_columns.py
@pytest.mark.parametrize("fx,fw,M,K,N", [
    (E4M3, E3M4, 2048, 2560, 640), (E4M3, E3M4, 300, 1152, 36), (E4M3, E2M5, 700, 500, 100), (E4M3, fpq.Format(5, 2, 16), 900, 386, 200),
    (E5M2, E3M4, 513, 700, 260), (E4M3, E2M1, 1300, 1540, 1000), (E4M3, E4M3, 2300, 900, 1030), (E5M2, E5M2, 1200, 1700, 1028),
    (E4M3, E1M2, 9217, 1300, 324), (E4M3, E3M4, 2048, 2560, 638), (E4M3, E3M4, 700, 640, 65), (E4M3, E3M4, 1111, 1300, 1283),
    (E4M3, E2M1, 3001, 1280, 1282), (E4M3, E4M3, 2100, 2560, 639)])
def test_linear_layers_on_pairs(fx, fw, M, K, N):
    assert fpq.fpq_linear_contraction(M, N, K, fx, fw) == PAIRS


@pytest.mark.parametrize("fx,fw,M,K,N,form", [
    (E4M3, E2M1, 8192, 320, 960, GENERAL), (E4M3, E2M1, 64, 5120, 320, FEW_ROWS), (E4M3, E3M4, 300, 640, 65, GENERAL),
    (E4M3, E2M1, 2, 1280, 1280, FEW_ROWS), (E4M3, E2M1, 8, 5120, 10240, FEW_ROWS), (E4M3, fpq.Format(6, 1, 31), 64, 64, 64, OTHER),
    (E5M2, E4M3, 64, 320, 320, FEW_ROWS), (E4M3, E1M2, 100, 640, 320, FEW_ROWS), (E4M3, E2M1, 127, 5120, 10240, GENERAL),
    (E4M3, E4M3, 127, 320, 320, FEW_ROWS), (E4M3, E4M3, 128, 320, 320, GENERAL), (E4M3, E4M3, 64, 322, 320, GENERAL),
    (E4M3, E4M3, 1, 96, 160, CUDA_CORES), (E4M3, E3M4, 8, 320, 320, GENERAL)])
def test_other_linear_layers(fx, fw, M, K, N, form):
    assert fpq.fpq_linear_contraction(M, N, K, fx, fw) == form


# test_gpu_pair_tiles.py
@pytest.mark.parametrize("B,C,H,W,Co,stride", [
    (2, 320, 64, 64, 320, 1), (2, 640, 32, 32, 640, 1), (64, 192, 32, 32, 192, 1), (8, 512, 32, 32, 512, 1), (3, 320, 45, 45, 324, 1),
    (5, 136, 30, 17, 100, 1), (50, 416, 11, 11, 608, 1), (2, 192, 7, 5, 288, 1), (1, 256, 13, 96, 70, 1), (16, 256, 32, 32, 256, 1),
    (9, 150, 7, 9, 104, 1), (3, 320, 45, 77, 320, 2), (2, 320, 64, 64, 320, 2), (13, 128, 9, 8, 100, 2), (1, 200, 7, 120, 256, 2),
    (1, 64, 3, 253, 72, 2), (40, 96, 4, 3, 72, 2), (9, 320, 31, 30, 640, 2), (24, 192, 48, 48, 320, 2), (3, 130, 25, 41, 96, 2),
    (7, 64, 11, 9, 72, 2)])
def test_convolutions_on_pairs(B, C, H, W, Co, stride):
    for fw in (E4M3, E2M1):
        assert fpq.fpq_conv2d_contraction(B, C, H, W, Co, 3, 3, 1, stride, E4M3, fw) == PAIRS


# the kernels for few rows under each policy: one with warp-level MMAs where the route may be one kernel, the one on the CUDA cores always
@pytest.mark.parametrize("M,K,N,alone,never", [(2, 1280, 1280, FEW_ROWS, CUDA_CORES), (64, 5120, 320, FEW_ROWS, GENERAL),
                                               (8, 5120, 10240, FEW_ROWS, GENERAL), (1, 4, 1, CUDA_CORES, CUDA_CORES)])
def test_few_rows_by_policy(M, K, N, alone, never):
    try:
        for policy, form in ((fpq.PATH_AUTO, alone), (fpq.PATH_FUSED, alone), (fpq.PATH_TWO_KERNELS, never),
                             (fpq.PATH_TWO_KERNELS_NARROW, never)):
            fpq.fpq_set_path_policy(policy)
            assert fpq.fpq_linear_contraction(M, N, K, E4M3, E2M1) == form
    finally:
        fpq.fpq_set_path_policy(fpq.PATH_AUTO)


# what measured faster (us, one kernel / two: 11.2 / 7.9, 8.0 / 6.2, 10.0 / 7.9, 7.4 / 6.2; 2.9 / 5.0, 3.7 / 5.2, 16 / 23, 8.1 / 9.9, 3.6 / 6.6, 6.8 / 8.2)
@pytest.mark.parametrize("M,K,N,form", [
    (24, 1024, 10240, GENERAL), (48, 512, 7680, GENERAL), (20, 1024, 10240, GENERAL), (48, 1024, 3840, GENERAL), (48, 64, 5120, FEW_ROWS),
    (120, 100, 1920, FEW_ROWS), (9, 5120, 10240, FEW_ROWS), (24, 1920, 5120, FEW_ROWS), (64, 1280, 640, FEW_ROWS), (112, 2560, 1280, FEW_ROWS)])
def test_few_rows_or_two_kernels(M, K, N, form):
    for fw in (E4M3, E2M1):
        assert fpq.fpq_linear_contraction(M, N, K, E4M3, fw) == form


def test_policies_and_errors():
    L = fpq.lib()
    try:
        fpq.fpq_set_path_policy(fpq.PATH_TWO_KERNELS_NARROW)
        assert fpq.fpq_linear_contraction(2048, 640, 2560, E4M3, E3M4) == GENERAL
        assert fpq.fpq_conv2d_contraction(2, 320, 64, 64, 320, 3, 3, 1, 1, E4M3, E2M1) == GENERAL
    finally:
        fpq.fpq_set_path_policy(fpq.PATH_AUTO)
    assert fpq.fpq_conv2d_contraction(2, 64, 8, 8, 64, 3, 3, 1, 1, E4M3, fpq.Format(6, 1, 31)) == OTHER
    assert fpq.fpq_linear_contraction(0, 640, 2560, E4M3, E3M4) == GENERAL
    assert L.fpq_linear_contraction(-1, 1, 1, E4M3.c(), E4M3.c()) == fpq.ERR_SHAPE
    assert L.fpq_linear_contraction(1, 1, 0, E4M3.c(), E4M3.c()) == fpq.ERR_SHAPE
    assert L.fpq_linear_contraction(1, 1, 1, fpq.Format(6, 3, 7).c(), E4M3.c()) == fpq.ERR_FORMAT
    assert L.fpq_conv2d_contraction(2, 0, 8, 8, 64, 3, 3, 1, 1, E4M3.c(), E4M3.c()) == fpq.ERR_SHAPE
    assert L.fpq_conv2d_contraction(2, 64, 1, 1, 64, 3, 3, 0, 1, E4M3.c(), E4M3.c()) == fpq.ERR_SHAPE
    assert L.fpq_conv2d_contraction(2, 64, 8, 8, 64, 3, 3, 1, 1, fpq.Format(6, 3, 7).c(), E4M3.c()) == fpq.ERR_FORMAT


# few outputs: what measured faster or within a few per cent of it (us, pairs / general, E2M1 weights: 320 -> 4 at 64 x 64, batch 2 11.9 / 11.6, with E4M3
# weights 11.8 / 13.7; 16 x 256 -> 32 at 32 x 32 10.8 / 11.8; 8 x 320 -> 32 at stride 2 17.1 / 19.6; 1280 -> 32 at 8 x 8 16.3 / 8.4; 1280
# -> 16 at 16 x 16 16.5 / 8.5; 320 -> 3 at 32 x 32 10.0 / 7.5; 15 x 992 -> 24 at 21 x 21 19.8 / 16.6; 1280 -> 32 at stride 2 15.4 / 9.8)
@pytest.mark.parametrize("B,C,H,W,Co,stride,form", [
    (2, 320, 64, 64, 4, 1, PAIRS), (16, 256, 32, 32, 32, 1, PAIRS), (8, 320, 64, 64, 32, 2, PAIRS), (28, 192, 10, 10, 16, 1, PAIRS),
    (2, 1280, 8, 8, 32, 1, GENERAL), (2, 1280, 8, 8, 4, 1, GENERAL), (2, 1280, 16, 16, 16, 1, GENERAL), (2, 320, 32, 32, 3, 1, GENERAL),
    (15, 992, 21, 21, 24, 1, GENERAL), (8, 640, 32, 32, 32, 1, GENERAL), (2, 1280, 16, 16, 32, 2, GENERAL), (1, 480, 27, 27, 24, 2, GENERAL),
    (2, 1280, 8, 8, 33, 1, GENERAL), (2, 320, 30, 30, 64, 1, GENERAL), (2, 352, 28, 28, 40, 1, GENERAL), (25, 320, 15, 15, 48, 1, PAIRS),
    (4, 1312, 61, 61, 64, 1, PAIRS), (4, 128, 59, 59, 8, 1, PAIRS)])
def test_convolutions_of_few_outputs(B, C, H, W, Co, stride, form):
    for fw in (E4M3, E2M1):
        assert fpq.fpq_conv2d_contraction(B, C, H, W, Co, 3, 3, 1, stride, E4M3, fw) == form


# windows whose taps do not go three to a load (16, 25, 49): a load per tap bounds the pairs (us, pairs / general: 4 x 348 -> 98 at
# 7 x 7, 25 taps 22.5 / 15.7; 271 -> 924 at 10 x 10 22.6 / 15.1; 14 x 631 -> 85 at 18 x 18 36.9 / 25.3; 331 -> 569 at 16 x 16, 16 taps 17.0 /
# 13.1; 22 x 107 -> 493 at 8 x 8 10.3 / 16.2; 22 x 55 -> 745 at 40 x 40 48.7 / 82.7; 4 x 249 -> 30 at 22 x 22, 49 taps 27.8 / 19.6)
@pytest.mark.parametrize("B,C,H,W,Co,R,form", [
    (4, 348, 7, 7, 98, 5, GENERAL), (1, 271, 10, 10, 924, 5, GENERAL), (14, 631, 18, 18, 85, 5, GENERAL), (2, 331, 16, 16, 569, 4, GENERAL),
    (22, 107, 8, 8, 493, 4, PAIRS), (22, 55, 40, 40, 745, 4, PAIRS), (4, 249, 22, 22, 30, 7, GENERAL)])
def test_large_windows(B, C, H, W, Co, R, form):
    for fw in (E4M3, E2M1):
        assert fpq.fpq_conv2d_contraction(B, C, H, W, Co, R, R, R // 2, 1, E4M3, fw) == form
