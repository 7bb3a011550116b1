"""The tensor-core scan against the byte-permute scan asked for by its lanes (the
default takes the tensor cores where queries share lists, so it is no
reference): candidate stores, ids and distances bit for bit, at the benchmark's
operating point and on the 10k x 128 configuration."""
import numpy as np
import pytest

from paper_2511_03298_gb300 import synth

from test_gpu_parity import gpu_index, small_index

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ksc():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    return ksc


def _same(a, b):
    return all(bool((x == y).all()) for x, y in zip(a, b))


def _compare(ksc, g, Q, P, R, tile=0):
    import torch
    tc, by = ksc.search_opts(scan_tc=True, tile_blocks=tile), ksc.search_opts(lanes_per_query=8)
    assert _same(g.search(Q, 10, P, R, opts=tc), g.search(Q, 10, P, R, opts=by))
    probes, _ = g.rank_lists(Q, P, want_scores=False)
    assert _same(g.search_with_probes(Q, probes, 10, R, opts=tc), g.search_with_probes(Q, probes, 10, R, opts=by))
    rng = np.random.default_rng(3)
    npb = torch.from_numpy(rng.integers(1, P + 1, len(Q)).astype(np.int32)).cuda()
    rr = torch.from_numpy(rng.integers(10, R + 1, len(Q)).astype(np.int32)).cuda()
    assert _same(*(g.search_varprobe(Q, 10, npb, rr, nprobe_max=P, rerank_max=R, opts=o) for o in (tc, by)))


@pytest.mark.parametrize("tile", [0, 4, 12])
def test_small_configuration(ksc, tile):
    import torch
    ix, Q = small_index("small")
    _compare(ksc, gpu_index(ksc, ix), torch.from_numpy(Q).cuda(), 12, 200, tile)


def test_full_size_workload(ksc):
    import torch
    X, Q = synth.base(2), synth.queries(2)
    g = ksc.build_index(torch.from_numpy(X).cuda(), 1024, 64, perm=synth.build_perm(2, len(X)))
    _compare(ksc, g, torch.from_numpy(Q).cuda(), 7, 200)


@pytest.mark.parametrize("M,ds", [(1, 4), (9, 1), (50, 2), (80, 1), (97, 1), (104, 1), (128, 1)])
@pytest.mark.parametrize("nq,P", [(16, 5), (17, 5), (700, 5), (600, 2)])
def test_subspaces_and_groups_asked_for(ksc, M, ds, nq, P):
    """The largest subspace counts hold 16 queries an item, and small batches take
    the tensor cores only when asked to."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(M + nq)
    X = torch.randn(20_000, M * ds, generator=g, device="cuda")
    ix = ksc.build_index(X, 40, M, iters=2)
    _compare(ksc, ix, torch.randn(nq, M * ds, generator=g, device="cuda"), P, 60)
