"""Where many queries of a batch share the lists, the filtered scan runs on the
tensor cores without being asked.  Its results are whole-number keys, so ids,
distances and candidate stores equal those of the byte-permute scan (asked for
by its lanes per query) bit for bit: over subspace counts around the 8 of an
operand chunk, up to the largest; query groups around 16, 64 and their
multiples; many items per thread block; tied and duplicated vectors, which fill
the per-warp key buffers and the candidate store.
"""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ksc():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    return ksc


def _case(ksc, n, d, L, M, nq, P, R, metric="l2", tile=0, distinct=0, cap=0):
    import torch
    g = torch.Generator().manual_seed(n + d + M)
    X = torch.randn(n, d, generator=g) + 2 * torch.randn(max(L // 2, 1), d, generator=g)[
        (torch.rand(n, generator=g) ** 2 * max(L // 2, 1)).long()]  # lists of unequal sizes
    if distinct:
        X = X[torch.randint(0, distinct, (n,), generator=g)].contiguous()
    Q = (X[torch.randint(0, n, (nq,), generator=g)] + 0.3 * torch.randn(nq, d, generator=g)).cuda()
    ix = ksc.build_index(X.cuda(), L, M, metric=metric, iters=3, seed=7)
    probes, _ = ix.rank_lists(Q, P, want_scores=False)
    a = ix.search_with_probes(Q, probes, 10, R, opts=ksc.search_opts(tile_blocks=tile, cand_cap=cap))
    assert ix.last_status() & ~1 == 0  # (1: a candidate store overflowed and was redone)
    b = ix.search_with_probes(Q, probes, 10, R, opts=ksc.search_opts(lanes_per_query=8, cand_cap=cap))
    assert all(torch.equal(x, y) for x, y in zip(a, b))
    # again on the same buffers (counters and item queues start over)
    c = ix.search_with_probes(Q, probes, 10, R, opts=ksc.search_opts(tile_blocks=tile, cand_cap=cap))
    assert all(torch.equal(x, y) for x, y in zip(a, c))


@pytest.mark.parametrize("M,ds", [(1, 4), (8, 2), (9, 1), (50, 2), (64, 2), (80, 1), (128, 1)])
def test_subspace_counts(ksc, M, ds):
    _case(ksc, 20_000, M * ds, 40, M, 700, 5, 60)


@pytest.mark.parametrize("nq", [600, 1600, 1700, 4100])
def test_query_groups(ksc, nq):
    _case(ksc, 14_000, 32, 50, 16, nq, 2, 25)


@pytest.mark.parametrize("tile", [4, 8, 2048])
def test_many_items(ksc, tile):
    _case(ksc, 250_000, 32, 48, 16, 3000, 9, 100, tile=tile)


@pytest.mark.parametrize("metric,distinct,cap", [("l2", 30, 0), ("ip", 0, 0), ("ip", 300, 128)])
def test_ties_and_full_buffers(ksc, metric, distinct, cap):
    _case(ksc, 12_000, 24, 32, 12, 1500, 6, 100, metric=metric, distinct=distinct, cap=cap)
