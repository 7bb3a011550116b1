"""Queries whose candidate store overflows: the R best of their recomputed keys,
gathered under the bound of the stored ones.  Same candidates as with a store
that holds everything, for stores of R keys (every pass recomputes), one more,
around the lists' sizes, and with duplicated vectors whose ties overflow the
gathered keys as well; few queries and many.
"""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq", [40, 700])
@pytest.mark.parametrize("R,cap", [(100, 100), (100, 101), (100, 512), (100, 1250), (1500, 1501), (1500, 2500)])
@pytest.mark.parametrize("metric,distinct", [("l2", 0), ("ip", 0), ("l2", 40)])
def test_overflowed_stores(metric, distinct, R, cap, nq):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    g = torch.Generator().manual_seed(2)
    sizes = [1249, 1250, 1251, 3000, 9000, 400, 20, 3830]  # lists by far-apart centres
    X = torch.cat([torch.randn(s, 16, generator=g) + 60 * torch.eye(16)[i] for i, s in enumerate(sizes)])
    X = X[torch.randperm(len(X), generator=g)].contiguous()
    if distinct:
        X = X[torch.randint(0, distinct, (len(X),), generator=g)].contiguous()
    Q = (X[torch.randint(0, len(X), (nq,), generator=g)] + 0.1 * torch.randn(nq, 16, generator=g)).cuda()
    ix = ksc.build_index(X.cuda(), 8, 8, metric=metric, iters=4, seed=3)
    probes, _ = ix.rank_lists(Q, 4, want_scores=False)
    a = ix.search_with_probes(Q, probes, 10, R, opts=ksc.search_opts(cand_cap=cap))
    assert ix.last_status() == ksc.STATUS_CAND_OVERFLOW and ix.search_stats()["overflow_queries"] > 0
    b = ix.search_with_probes(Q, probes, 10, R, opts=ksc.search_opts(cand_cap=40_000))
    assert ix.last_status() == 0
    assert all(torch.equal(x, y) for x, y in zip(a, b))
