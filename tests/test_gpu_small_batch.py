"""Searches of a few queries (a cluster per query through ranking, tables and
scan items, a CTA per query through selection and re-rank) against the oracle:
candidate keys bit-exact with given probes, and results equal to the same
queries inside a large batch (the general kernels), over batch sizes, probe
counts around the kernels' chunks, subspace widths, candidate counts around the
selections' limits, per-query settings, small candidate stores (overflow) and
tied distances.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    return torch, ksc


def _data(n, d, seed, kind="float"):
    rng = np.random.default_rng(seed)
    c = rng.uniform(-4, 4, size=(24, d))
    X = c[rng.integers(0, 24, n)] + rng.normal(size=(n, d))
    Q = c[rng.integers(0, 24, 1600)] + rng.normal(size=(1600, d))
    if kind == "bytes":
        X, Q = (np.clip(np.rint(128 + 20 * a), 0, 255) for a in (X, Q))
    if kind == "ties":  # few distinct rows: long runs of equal distances
        X = np.rint(X[rng.integers(0, 40, n)])
    return X.astype(np.float32), Q.astype(np.float32)


@pytest.mark.parametrize("d,M,metric,kind,L", [(32, 16, "l2", "float", 37), (60, 15, "l2", "bytes", 64), (48, 48, "ip", "float", 50),
                                               (24, 3, "l2", "float", 20), (130, 65, "l2", "float", 33), (64, 32, "l2", "ties", 40),
                                               (256, 128, "ip", "float", 18), (520, 130, "l2", "float", 12)])
def test_equal_to_large_batch(env, d, M, metric, kind, L):
    torch, ksc = env
    X, Q = _data(6000, d, d + M, kind)
    ix = ksc.build_index(torch.from_numpy(X).cuda(), L, M, metric=metric, iters=3, seed=3)
    Qd = torch.from_numpy(Q).cuda()
    for P, R, k in ((1, 30, 10), (min(L, 7), 200, 10), (L, 513, 40), (min(L, 9), 700, 700), (min(L, 12), 64, 64)):
        ref = ix.search(Qd, k, P, R)  # 1600 queries: the general kernels
        for b in (1, 3, 64, 303):
            got = ix.search(Qd[:b].contiguous(), k, P, R)
            assert torch.equal(got[0], ref[0][:b]) and torch.equal(got[1], ref[1][:b]), (P, R, k, b)
    # per-query settings
    g = torch.Generator(device="cuda").manual_seed(1)
    P = torch.randint(1, min(L, 11) + 1, (1600,), generator=g, device="cuda", dtype=torch.int32)
    R = torch.randint(20, 150, (1600,), generator=g, device="cuda", dtype=torch.int32)
    ref = ix.search_varprobe(Qd, 10, P, R, min(L, 11), 150)
    got = ix.search_varprobe(Qd[:50].contiguous(), 10, P[:50].contiguous(), R[:50].contiguous(), min(L, 11), 150)
    assert torch.equal(got[0], ref[0][:50]) and torch.equal(got[1], ref[1][:50])
    # a store too small for the unfiltered part and for the rest: redone exactly
    opts = ksc.search_opts(cand_cap=R_SMALL)
    ref = ix.search(Qd, 10, min(L, 9), R_SMALL)
    got = ix.search(Qd[:40].contiguous(), 10, min(L, 9), R_SMALL, opts=opts)
    assert torch.equal(got[0], ref[0][:40]) and torch.equal(got[1], ref[1][:40])


R_SMALL = 25


@pytest.mark.parametrize("nq,P,R,cap", [(1, 5, 60, 0), (2, 1, 600, 0), (40, 29, 100, 0), (40, 29, 100, 150),
                                        (7, 60, 1500, 0), (200, 13, 33, 0), (1, 60, 20, 40)])
def test_candidates_bit_exact(env, nq, P, R, cap):
    torch, ksc = env
    X, Q = _data(9000, 32, 5)
    ix = oracle.build_index(X, 60, 16, False, np.random.default_rng(2).permutation(9000).astype(np.int64), iters=2)
    gi = ksc.index_import(ix)
    Q = Q[:nq]
    probes = np.stack([oracle.rank(q, ix["c_rank"], False, P)[0] for q in Q]).astype(np.int32)
    if P > 20:  # an unused slot in the middle
        probes[:, 11] = -1
    opts = ksc.search_opts(cand_cap=cap) if cap else None
    _, _, cand, ncand = gi.search_with_probes(torch.from_numpy(Q).cuda(), torch.from_numpy(probes).cuda(), 10, R, opts=opts)
    cand, ncand = cand.cpu().numpy().view(np.uint64), ncand.cpu().numpy()
    for i in range(nq):
        pr = probes[i][probes[i] >= 0]
        Ql, b, _ = oracle.lut_q8(Q[i], ix, pr)
        ref = oracle.scan_topr(ix, pr, Ql, b, R)
        assert ncand[i] == len(ref)
        assert np.array_equal(cand[i, :len(ref)], ref), i


def test_large_nlist_and_lists(env):
    """Probes past one chunk of the item kernel and lists above the fused ranking's limit."""
    torch, ksc = env
    rng = np.random.default_rng(8)
    X = rng.normal(size=(30000, 16)).astype(np.float32)
    Q = rng.normal(size=(1400, 16)).astype(np.float32)
    ix = ksc.build_index(torch.from_numpy(X).cuda(), 9000, 8, iters=1, seed=1)
    Qd = torch.from_numpy(Q).cuda()
    for P in (600, 1024):
        ref = ix.search(Qd, 10, P, 200)
        got = ix.search(Qd[:20].contiguous(), 10, P, 200)
        assert torch.equal(got[0], ref[0][:20]) and torch.equal(got[1], ref[1][:20])
