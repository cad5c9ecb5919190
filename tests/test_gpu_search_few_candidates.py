"""The search with few candidates on tensors of many blocks: the blocks' sums are shared by the last kernel's threads; counts of
candidates that divide them and that do not, from one to all of them."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2408_06995_b200 as fpq

pytestmark = pytest.mark.gpu

ENC = O.FP8_ENCODINGS + O.FP4_ENCODINGS


@pytest.mark.parametrize("n,n_enc,n_clip", [(4096, 1, 1), (300001, 1, 1), (1 << 20, 2, 1), (700003, 3, 1), (150000, 4, 7), (100000, 5, 17),
                                            (40000, 4, 128), (30000, 3, 171), (30000, 6, 170)])
def test_matches_the_oracle(n, n_enc, n_clip):
    x = np.random.default_rng(n).standard_normal(n).astype(np.float32)
    encs = ENC[:n_enc]
    clips = fpq.fpq_search_clip_candidates(float(np.abs(x).max()), n_clip)
    mse, best = fpq.fpq_search_format(torch.from_numpy(x).cuda(), [fpq.Format(f.e, f.m, f.B, fpq.SAT_PAPER) for f in encs], clips.cuda())
    assert fpq.fpq_read_status() == fpq.OK
    got = mse.cpu().numpy()
    # (the bound of test_gpu_search.py: FP32 sums of 512 squared errors, then double)
    np.testing.assert_allclose(got, O.search_mse(x, encs, clips.numpy()), rtol=2e-6, atol=0)
    assert tuple(best.cpu().numpy()) == O.select_encoding_and_bias(got)
    again, _ = fpq.fpq_search_format(torch.from_numpy(x).cuda(), [fpq.Format(f.e, f.m, f.B, fpq.SAT_PAPER) for f in encs], clips.cuda())
    assert torch.equal(mse, again)
