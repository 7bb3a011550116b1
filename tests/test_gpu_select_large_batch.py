"""Threshold and selection of 257 to 512 candidates by warps in batches that give
every SM 32 of them, by CTAs below: both give the candidates of a sort of all
keys of the probed lists."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [257, 400, 512])
def test_candidates(R):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    g = torch.Generator(device="cuda").manual_seed(R)
    n_q = 32 * torch.cuda.get_device_properties(0).multi_processor_count
    X = torch.randn(20_000, 16, generator=g, device="cuda")
    Q = torch.randn(n_q + 40, 16, generator=g, device="cuda")
    ix = ksc.build_index(X, 40, 8, iters=2)
    probes, _ = ix.rank_lists(Q, 5, want_scores=False)
    # every key of the probed lists: R beyond their number
    full, nf = ix.search_with_probes(Q[:300].contiguous(), probes[:300].contiguous(), 10, 4096,
                                     opts=ksc.search_opts(cand_cap=8192))[2:]
    assert (nf < 4096).all()
    for nq in (n_q - 1, n_q, n_q + 40):
        ids, dists, cand, n = ix.search_with_probes(Q[:nq].contiguous(), probes[:nq].contiguous(), 10, R)
        assert ix.last_status() == 0
        m = torch.clamp(nf, max=R)
        assert torch.equal(n[:300], m)
        ok = torch.arange(R, device="cuda")[None] < m[:, None]
        assert torch.equal(torch.where(ok, cand[:300], 0), torch.where(ok, full[:, :R], 0))
