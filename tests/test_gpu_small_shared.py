"""Batches just below the small-batch kernels' limit take the general ones where
their queries share the lists (told by the number of launches), and the small
ones where they do not; results equal those of the same queries in a large
batch on both sides."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,nq,P,small", [(64, 303, 2, False), (64, 250, 16, False), (64, 200, 16, True),
                                          (1024, 303, 3, True), (1024, 303, 4, False), (1024, 250, 8, True),
                                          (1024, 250, 9, False), (1024, 150, 64, True), (1024, 1, 1024, True)])
def test_shared_lists_take_the_general_path(L, nq, P, small):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    g = torch.Generator(device="cuda").manual_seed(L)
    X = torch.randn(30_000, 32, generator=g, device="cuda")
    Q = torch.randn(700, 32, generator=g, device="cuda")
    ix = ksc.build_index(X, L, 16, iters=2)
    q = Q[:nq].contiguous()
    ref = ix.search(Q, 10, P, 100)
    ix.profile(True)
    got = ix.search(q, 10, P, 100)
    _, launches = ix.profile_read()
    ix.profile(False)
    # small: at most 3 launches of ranking, then tables, scan, threshold, scan, selection and re-rank
    print("launches", launches)
    assert (launches <= 8) == small, launches
    assert torch.equal(got[0], ref[0][:nq]) and torch.equal(got[1], ref[1][:nq])
