"""Index construction's tensor-core assignment and register codebook kernels
against plain FP64 torch: lists and codes equal up to FP32 near-ties, at the
edges of tiles (rows around 128, centroids around 256, dimensions around 64),
at every sub-vector width the kernels serve and on data that the FP16 operands'
bound separates badly (a large common offset, duplicated centroids, tiny and
huge scales) or not at all (the FP32 kernel).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ksc():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    return ksc


def _check(ksc, X, L, M, metric="l2", iters=3):
    import torch
    ix = ksc.build_index(torch.from_numpy(X).cuda(), L, M, metric=metric, iters=iters, seed=7)
    e = ix.export(fields=("c_rank", "c_mean", "codebook", "codes", "assign"))
    x, c = torch.from_numpy(X).double(), torch.from_numpy(e["c_rank"]).double()
    dot = x @ c.T
    s = -dot if metric == "ip" else (c * c).sum(1) - 2 * dot
    a = torch.from_numpy(e["assign"]).long()
    n, d = X.shape
    # FP32 rule: sum of d products and one more rounding, each 2^-24 of |x| |c| at most
    size = x.norm(dim=1) * c.norm(dim=1).max()
    tol = 2 * (d + 2) * 2.0 ** -24 * (2 * size + c.norm(dim=1).max() ** 2)
    assert (s.gather(1, a[:, None])[:, 0] <= s.min(1).values + tol).all()
    # codes: nearest codeword of the residual (FP32 subtraction), up to its FP32 sum
    cm = torch.from_numpy(e["c_mean"])
    R = (torch.from_numpy(X) - cm[a]).double().view(n, M, d // M)
    cb = torch.from_numpy(e["codebook"]).double()
    D = (R[:, :, None] - cb[None]).square().sum(3)
    got = D.gather(2, torch.from_numpy(e["codes"]).long()[:, :, None])[:, :, 0]
    best = D.min(2).values
    # FP32: the differences round by 2^-24 of |r| + |w|, the squares and sums by (ds + 1) 2^-24 of the sum
    ds = d // M
    tol = 2 * (ds + 3) * 2.0 ** -24 * (R.abs().amax(2) + cb.abs().amax()) ** 2 * ds
    assert (got <= best + tol).all()
    # the mean centroids are the FP64 means of the lists
    for p in range(0, L, max(1, L // 20)):
        m = a == p
        if m.any():
            ref = x[m].mean(0)
            assert (cm[p].double() - ref).abs().max() <= 2.0 ** -23 * x[m].abs().max()
    return e


@pytest.mark.parametrize("n,d,L,M", [(127, 16, 3, 16), (128, 64, 255, 32), (129, 65, 7, 65), (1500, 63, 256, 21),
                                     (1500, 128, 257, 32), (3000, 192, 600, 24), (2000, 320, 64, 64),
                                     (2000, 784, 40, 196), (1200, 24, 30, 3), (900, 10, 20, 2), (600, 1024, 33, 128)])
@pytest.mark.parametrize("metric", ["l2", "ip"])
def test_tile_edges(ksc, n, d, L, M, metric):
    rng = np.random.default_rng(n + d + L)
    L = min(L, n)
    X = (rng.uniform(-3, 3, size=(20, d))[rng.integers(0, 20, n)] + rng.normal(size=(n, d))).astype(np.float32)
    _check(ksc, X, L, M, metric)


@pytest.mark.parametrize("kind", ["offset", "duplicates", "tiny", "huge", "fp32_range", "zeros", "mixed"])
def test_hard_data(ksc, kind):
    rng = np.random.default_rng(11)
    X = rng.normal(size=(1500, 32)).astype(np.float32)
    if kind == "offset":  # every centroid is inside the bound: rows go to the FP32 kernel
        X += np.float32(300.0)
    elif kind == "duplicates":  # equal centroids: ties to the lower id
        X = np.repeat(X[:50], 30, axis=0)
    elif kind == "tiny":
        X *= np.float32(1e-9)
    elif kind == "huge":
        X *= np.float32(1e12)
    elif kind == "fp32_range":  # outside the operands' range: FP32 throughout
        X *= np.float32(1e16)
    elif kind == "zeros":
        X[:] = 0
    else:  # dimensions of very different scale
        X *= np.logspace(-6, 3, 32).astype(np.float32)
    e = _check(ksc, X, 40, 16)
    if kind == "duplicates":
        c = e["c_rank"]
        for p, q in zip(*np.nonzero((c[:, None] == c[None]).all(2))):
            if p < q:
                assert not (e["assign"] == q).any()
