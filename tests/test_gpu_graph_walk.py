"""The graph walk's register-resident result set (hybrid search, Sec. 4.4) at
its edges: capacities around multiples of 32 (one to three entries per lane),
subspace counts around multiples of 32 (one to eight tables per lane) and lists
shorter than a walk.  Candidate keys bit-exact against the oracle's walk.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,dsub,efs,tau,L", [
    (32, 1, 31, 1 << 20, 8), (33, 1, 32, 1 << 20, 8), (33, 1, 33, 6, 8), (64, 1, 64, 1 << 20, 8),
    (65, 1, 65, 1 << 20, 8), (40, 2, 95, 20, 8), (129, 1, 96, 1 << 20, 8), (16, 2, 1, 1 << 20, 8),
    (16, 2, 96, 1 << 20, 60), (16, 2, 64, 1 << 20, 400)])
def test_walk_bit_exact(M, dsub, efs, tau, L):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    n, d, nq, P, R, k = 2400, M * dsub, 12, 6, 90, 10
    rng = np.random.default_rng(1000 * M + efs)
    centres = rng.uniform(-3, 3, size=(6, d))
    X = (centres[rng.integers(0, 6, n)] + rng.normal(size=(n, d))).astype(np.float32)
    Q = (centres[rng.integers(0, 6, nq)] + rng.normal(size=(nq, d))).astype(np.float32)
    ix = oracle.build_index(X, L, M, False, rng.permutation(n).astype(np.int64), iters=2)
    g, entry = oracle.build_graph(ix)
    gi = ksc.index_import(dict(ix, graph=g, entry=entry))
    probes = np.stack([oracle.rank(q, ix["c_rank"], False, P)[0] for q in Q]).astype(np.int32)
    opts = ksc.search_opts(hybrid=True, n_near=1, efs=efs, tau=tau)
    ids, dists, cand, ncand = gi.search_with_probes(torch.from_numpy(Q).cuda(), torch.from_numpy(probes).cuda(), k, R,
                                                    opts=opts)
    cand, ncand = cand.cpu().numpy().view(np.uint64), ncand.cpu().numpy()
    for qi in range(nq):
        Ql, b, _ = oracle.lut_q8(Q[qi], ix, probes[qi])
        ref, _ = oracle.hybrid_topr(ix, g, entry, probes[qi], Ql, b, R, n_near=1, efs=efs, tau=tau)
        assert ncand[qi] == len(ref), qi
        assert np.array_equal(cand[qi, :len(ref)], ref), qi
