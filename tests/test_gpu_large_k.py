"""The CTA re-ranks' order of more than 256 results (sorted in shared memory; up to
256 counted): around 256, 512 and a power of two, with as many candidates, more and
fewer than k, FP32 and exact U8 rows, L2 and inner products, small and larger
batches.  Byte-valued data: distances are whole numbers, the order of (distance,
id) is known."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq", [5, 330])
@pytest.mark.parametrize("k,R", [(10, 256), (10, 257), (256, 300), (257, 257), (300, 600), (512, 600), (513, 513), (513, 2000), (1000, 1000), (1024, 1024), (1024, 4096)])
@pytest.mark.parametrize("metric,band", [("l2", 0), ("l2", -1), ("ip", 0)])
def test_order(nq, k, R, metric, band):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    rng = np.random.default_rng(k + R)
    X = rng.integers(0, 256, size=(8000, 32)).astype(np.float32)
    Q = rng.integers(0, 256, size=(nq, 32)).astype(np.float32)
    ix = ksc.build_index(torch.from_numpy(X).cuda(), 16, 16, metric=metric, iters=3, seed=1)
    opts = ksc.search_opts(rerank_band=band)
    Qd = torch.from_numpy(Q).cuda()
    for P in (1, 9):
        probes, _ = ix.rank_lists(Qd, P, want_scores=False)
        cand = ix.search_with_probes(Qd, probes, k, R, opts=opts)[2].cpu().numpy().view(np.uint64)
        ids, dists = (v.cpu().numpy() for v in ix.search(Qd, k, P, R, opts=opts))
        for q in range(nq):
            c = (cand[q][cand[q] != np.uint64(0xffffffffffffffff)] & np.uint64(0xffffffff)).astype(np.int64)
            D = np.square(X[c] - Q[q]).sum(1) if metric == "l2" else -(X[c] @ Q[q])  # whole numbers below 2^24
            order = np.lexsort((c, D))[:k]
            n = len(order)
            np.testing.assert_array_equal(ids[q, :n], c[order])
            np.testing.assert_array_equal(dists[q, :n], D[order] if metric == "l2" else -D[order])
            assert (ids[q, n:] == -1).all() and np.isinf(dists[q, n:]).all()
