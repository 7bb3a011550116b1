"""Probes given by the caller that name a list twice: its members are candidates
twice, equal keys that the CTA re-ranks still have to place one by one (every
slot written).  Small and larger batches, k on both sides of 32, R on both sides
of the counted order, FP32 and exact U8 rows (byte-valued data: distances are
whole numbers, so the order of (distance, id) is known exactly)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq", [16, 400])
@pytest.mark.parametrize("k,R", [(10, 200), (64, 200), (64, 700), (700, 700)])
@pytest.mark.parametrize("band", [0, -1])
def test_repeated_lists(nq, k, R, band):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    rng = np.random.default_rng(k + R)
    X = rng.integers(0, 256, size=(6000, 32)).astype(np.float32)
    Q = rng.integers(0, 256, size=(nq, 32)).astype(np.float32)
    ix = ksc.build_index(torch.from_numpy(X).cuda(), 16, 16, iters=3, seed=1)
    probes = np.stack([rng.permutation(16)[[0, 1, 0, 2, 1]] for _ in range(nq)]).astype(np.int32)
    Qd, Pd = torch.from_numpy(Q).cuda(), torch.from_numpy(probes).cuda()
    opts = ksc.search_opts(rerank_band=band)
    for want in (True, False):
        # freed blocks of the outputs' sizes: a slot left unwritten shows them
        junk = [torch.full((nq, k), -77, dtype=torch.int64, device="cuda"), torch.full((nq, k), -77.0, device="cuda")]
        del junk
        ids, dists, cand, _ = ix.search_with_probes(Qd, Pd, k, R, want_cands=want, opts=opts)
        if want:
            keys = cand.cpu().numpy().view(np.uint64)
        ids, dists = ids.cpu().numpy(), dists.cpu().numpy()
        repeats = 0
        for q in range(nq):
            c = (keys[q][keys[q] != np.uint64(0xffffffffffffffff)] & np.uint64(0xffffffff)).astype(np.int64)
            repeats += len(c) - len(np.unique(c))
            D = np.square(X[c] - Q[q]).sum(1)  # whole numbers below 2^24
            order = np.lexsort((c, D))[:k]
            n = len(order)
            np.testing.assert_array_equal(ids[q, :n], c[order])
            np.testing.assert_array_equal(dists[q, :n], D[order])
            assert (ids[q, n:] == -1).all() and np.isinf(dists[q, n:]).all()
        assert repeats > 0
