"""The fused tables with more threads per block (large tables: many subspaces,
probes or wide rows), for a batch, against the same queries searched a few at a
time, whose tables another kernel computes: the candidates' whole-number keys are
equal.  Fewer rows than threads, steps of the row walk above and below the
subspace count, dimensions above and below the thread count, per-query probes.
"""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,ds,P", [(196, 4, 4), (50, 2, 40), (128, 1, 24), (75, 8, 6), (256, 2, 3), (13, 3, 60)])
@pytest.mark.parametrize("metric", ["l2", "ip"])
def test_fused_tables_of_a_batch(metric, M, ds, P):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    g = torch.Generator().manual_seed(M)
    X = torch.randn(6000, M * ds, generator=g)
    Q = torch.randn(610, M * ds, generator=g).cuda()
    ix = ksc.build_index(X.cuda(), 64, M, metric=metric, iters=2, seed=1)
    probes, _ = ix.rank_lists(Q, P, want_scores=False)
    a = ix.search_with_probes(Q, probes, 10, 50)
    few = [ix.search_with_probes(Q[i:i + 61].contiguous(), probes[i:i + 61].contiguous(), 10, 50)
           for i in range(0, 610, 61)]
    for x, parts in zip(a, zip(*few)):
        assert torch.equal(x, torch.cat(parts))
    npb = (torch.arange(610, dtype=torch.int32) % P + 1).cuda()
    rr = torch.full_like(npb, 50)
    v = ix.search_varprobe(Q, 10, npb, rr, nprobe_max=P, rerank_max=50)
    few = [ix.search_varprobe(Q[i:i + 61].contiguous(), 10, npb[i:i + 61].contiguous(), rr[i:i + 61].contiguous(),
                              nprobe_max=P, rerank_max=50) for i in range(0, 610, 61)]
    for x, parts in zip(v, zip(*few)):
        assert torch.equal(x, torch.cat(parts))
