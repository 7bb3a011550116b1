"""The threshold and selection kernels with their keys in registers, at the sizes
where they change: as many near keys as they hold (2048, 4096, 8192), one more,
R keys exactly, fewer, and ties; in batches of every launch size.  The candidate
keys equal a sort of all keys of the probed lists (a store that holds everything,
R as large as it takes).
"""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq", [3, 310, 1300])
@pytest.mark.parametrize("size", [499, 500, 501, 1024, 2047, 2048, 2049, 4096, 4097, 8191, 8193])
@pytest.mark.parametrize("distinct", [0, 60])
def test_candidates_at_the_register_limits(nq, size, distinct):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    g = torch.Generator().manual_seed(size)
    R = 500
    sizes = [size, size, 700]
    X = torch.cat([torch.randn(s, 8, generator=g) + 90 * torch.eye(8)[i] for i, s in enumerate(sizes)])
    if distinct:
        X = torch.cat([p[torch.randint(0, distinct, (len(p),), generator=g)] for p in X.split(sizes)])
    Q = (X[torch.randint(0, len(X), (nq,), generator=g)] + 0.1 * torch.randn(nq, 8, generator=g)).cuda()
    ix = ksc.build_index(X.cuda(), 3, 4, iters=6, seed=2)
    probes, _ = ix.rank_lists(Q, 2, want_scores=False)
    _, _, cand, n = ix.search_with_probes(Q, probes, 10, R, opts=ksc.search_opts(cand_cap=20_000))
    assert ix.last_status() == 0
    # every key of the probed lists: R beyond their number
    _, _, full, nf = ix.search_with_probes(Q[:310].contiguous(), probes[:310].contiguous(), 10, 4096,
                                           opts=ksc.search_opts(cand_cap=20_000))
    m = torch.clamp(nf, max=R)
    assert torch.equal(n[:310], m)
    ok = torch.arange(R, device="cuda")[None] < m[:, None]
    assert torch.equal(torch.where(ok, cand[:310], 0), torch.where(ok, full[:, :R], 0))
