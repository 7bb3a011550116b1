"""The exact U8 re-rank asked for (its copies made at once) equal bit for bit to the
all-FP32 one, also for searches too small to make the copies by themselves."""
import numpy as np
import pytest

import test_gpu_rerank_low as low

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,M,k,R,P", [(144, 36, 10, 60, 3), (160, 40, 50, 51, 1), (256, 64, 10, 11, 2),
                                       (32, 16, 40, 300, 4), (128, 32, 64, 257, 8)])
@pytest.mark.parametrize("ints", [False, True])
def test_equal_fp32(d, M, k, R, P, ints):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    X, Q = low._data(6000, 310, d, d + k)
    Q = np.rint(Q) if ints else Q
    X[4000:4040] = X[:40]  # ties
    ix = ksc.build_index(torch.from_numpy(X).cuda(), 16, M, iters=2, seed=1)
    Qd = torch.from_numpy(Q).cuda()
    a = ix.search(Qd, k, P, R, opts=ksc.search_opts(rerank_band=1))
    b = ix.search(Qd, k, P, R, opts=ksc.search_opts(rerank_band=-1))
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
