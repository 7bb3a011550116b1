"""Re-ranks that read low-precision rows first: the exact U8 pass (byte-valued
rows past the warp kernel's range: wide rows, many neighbours, many candidates)
equal bit for bit to the all-FP32 re-rank, and the BF16 / FP8 shortlist within
its format's rounding, over widths that are and are not multiples of the vector
loads; the table rows of width 4 and the tensor-core preselection of wide rows
against the oracle.
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


def _data(n, nq, d, seed):
    rng = np.random.default_rng(seed)
    c = rng.uniform(30, 220, size=(16, d))
    X = np.clip(np.rint(c[rng.integers(0, 16, n)] + 12 * rng.normal(size=(n, d))), 0, 255).astype(np.float32)
    Q = (c[rng.integers(0, 16, nq)] + 12 * rng.normal(size=(nq, d))).astype(np.float32)
    return X, Q


@pytest.mark.parametrize("d,M,k,R,P", [(784, 196, 10, 200, 4), (144, 36, 10, 60, 3), (1024, 128, 1, 700, 6),
                                       (64, 32, 100, 400, 6), (128, 32, 33, 1500, 16), (160, 40, 50, 51, 1),
                                       (16, 4, 600, 1200, 9), (272, 68, 700, 900, 2), (132, 33, 10, 100, 4)])
@pytest.mark.parametrize("ints", [False, True])
def test_u8_rows_equal_fp32(env, d, M, k, R, P, ints):
    torch, ksc = env
    X, Q = _data(6000, 700, d, d + k)
    Q = np.rint(Q) if ints else Q
    X[4000:4040] = X[:40]  # ties
    ix = ksc.build_index(torch.from_numpy(X).cuda(), 16, M, iters=2, seed=1)
    Qd = torch.from_numpy(Q).cuda()
    a = ix.search(Qd, k, P, R)
    b = ix.search(Qd, k, P, R, opts=ksc.search_opts(rerank_band=-1))
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


@pytest.mark.parametrize("d,M", [(100, 50), (30, 15), (33, 11), (260, 65), (128, 32)])
@pytest.mark.parametrize("metric", ["l2", "ip"])
@pytest.mark.parametrize("prec", [1, 2])
def test_shortlist(env, d, M, metric, prec):
    torch, ksc = env
    rng = np.random.default_rng(d)
    X = rng.normal(size=(5000, d)).astype(np.float32)
    Q = rng.normal(size=(310, d)).astype(np.float32)
    ix = ksc.build_index(torch.from_numpy(X).cuda(), 8, M, metric=metric, iters=2, seed=1)
    Qd, R, Rf, k = torch.from_numpy(Q).cuda(), 300, 60, 60
    wide = ix.search(Qd, R, 8, R, opts=ksc.search_opts(rerank_band=-1))  # every candidate by FP32 distance
    got = ix.search(Qd, k, 8, R, opts=ksc.search_opts(precision=prec, rerank_final=Rf))
    low = ix.pair_distances(Qd, wide[0], prec)  # the candidates' low-precision distances
    low = -low if metric == "ip" else low
    cut = low.sort(1).values[:, Rf - 1:Rf]
    # the shortlist is the Rf best by that distance, up to FP32 summation order
    # ((d + 8) roundings of 2^-24 of the sum of magnitudes)
    mag = Qd.norm(dim=1) * torch.from_numpy(X).norm(dim=1).max().item() if metric == "ip" else \
        (Qd.norm(dim=1) + torch.from_numpy(X).norm(dim=1).max().item()).square()
    tol = 2 * (d + 8) * 2.0 ** -24 * 1.2 * mag[:, None]
    pos = (wide[0][:, :, None] == got[0][:, None, :])
    assert pos.any(1).all()  # every result is a candidate
    taken = pos.any(2)
    assert ((low <= cut + tol) | ~taken).all() and ((low >= cut - tol) | taken).all()
    # and they come by FP32 distance
    assert torch.equal(got[1], torch.where(taken, wide[1], torch.nan).nan_to_num(float("inf" if metric == "l2" else "-inf"))
                       .sort(1, descending=metric == "ip").values[:, :k])


@pytest.mark.parametrize("d,M,metric", [(784, 196, "l2"), (260, 65, "ip"), (1000, 250, "l2"), (320, 80, "ip"), (64, 16, "l2")])
def test_wide_ranking_and_tables(env, d, M, metric):
    """Lists ranked by the oracle's scores (FP32 near-ties aside), tables bit-exact."""
    torch, ksc = env
    X, Q = _data(3000, 1300, d, d)
    X, Q = (X - 120) / 50, (Q - 120) / 50
    ix = ksc.build_index(torch.from_numpy(X).cuda(), 40, M, metric=metric, iters=2, seed=1)
    e = ix.export()
    Qd = torch.from_numpy(Q).cuda()
    for nq in (1300, 5):
        probes, scores = ix.rank_lists(Qd[:nq].contiguous(), 12)
        q, c = torch.from_numpy(Q[:nq]).double(), torch.from_numpy(e["c_rank"]).double()
        s = -(q @ c.T) if metric == "ip" else torch.cdist(q, c).square()
        ref = s.gather(1, probes.cpu().long())
        best = s.sort(1).values[:, :12]
        assert ((ref - best).abs() <= 1e-4 * best.abs().clamp(min=1.0)).all()
        assert ((scores.cpu().double() - ref).abs() <= 1e-4 * ref.abs().clamp(min=1.0)).all()
    oi = oracle.make_index(e["X"], e["c_rank"], e["c_mean"], e["codebook"], e["codes"], e["assign"], ip=metric == "ip",
                           spherical=metric == "ip")
    pr = probes.cpu().numpy()
    lut, bias, scale = ix.compute_luts(Qd[:5].contiguous(), probes)
    for i in range(5):
        Ql, b, a = oracle.lut_q8(Q[i], oi, pr[i])
        assert np.array_equal(lut[i].cpu().numpy(), Ql.reshape(lut[i].shape)) and np.array_equal(bias[i].cpu().numpy(), b)
    # misaligned queries and a large batch (the fused kernel) give the same results
    buf = torch.empty(Qd.numel() + 1, device="cuda")
    off = buf[1:].view(Qd.shape)
    off.copy_(Qd)
    a, b = ix.search(Qd, 10, 6, 80), ix.search(off, 10, 6, 80)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
