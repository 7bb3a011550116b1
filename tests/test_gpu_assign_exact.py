"""The build's assignment against the FP32 rule restated exactly: score = ||c||^2 -
2 <x, c> (or -<x, c>), dot products and norms by FMAs over ascending
dimensions, the smallest score, ties to the lower list.  On both sides of the
rule that picks the tensor cores: tile edges of rows, lists and dimensions there,
data that leaves most rows to the FP32 kernels (more than 2048 of them), and
more rows than one pass takes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _fma(torch, a, b, c):
    """fl32(a b + c) of FP32 tensors: the FP64 sum rounded to odd, then to FP32."""
    p = a.double() * b.double()  # exact
    c = c.double()
    s = p + c
    t = s - p
    err = (p - (s - t)) + (c - t)
    bits = s.view(torch.int64)
    fix = (err != 0) & (bits & 1 == 0)
    return (bits + torch.where(fix, torch.where((err > 0) == (s > 0), 1, -1), 0)).view(torch.float64).float()


def _rule(torch, X, C, spherical):
    L, d = C.shape
    cn = torch.zeros(L, device="cuda")
    for t in range(d):
        cn = _fma(torch, C[:, t], C[:, t], cn)
    out = torch.empty(len(X), dtype=torch.int64, device="cuda")
    ids = torch.arange(L, device="cuda")
    step = max(1, (1 << 23) // L)
    for b in range(0, len(X), step):
        x = X[b:b + step]
        acc = torch.zeros((len(x), L), device="cuda")
        for t in range(d):
            acc = _fma(torch, x[:, t, None], C[None, :, t], acc)
        s = -acc if spherical else _fma(torch, torch.full_like(acc, -2.0), acc, cn[None].expand_as(acc))
        out[b:b + step] = torch.where(s == s.min(1, keepdim=True).values, ids, L).min(1).values
    return out


def _check(X, L, M, metric, iters=1):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    ix = ksc.build_index(X, L, M, metric=metric, iters=iters, seed=7)
    e = ix.export(fields=("c_rank", "assign"))
    want = _rule(torch, X, torch.from_numpy(e["c_rank"]).cuda(), metric == "ip")
    np.testing.assert_array_equal(e["assign"], want.cpu().numpy())


def _data(n, d, seed):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    mu = 6 * torch.rand((40, d), generator=g, device="cuda") - 3
    return mu[torch.randint(0, 40, (n,), generator=g, device="cuda")] + torch.randn((n, d), generator=g, device="cuda")


@pytest.mark.parametrize("n,d,L,M", [(20_001, 65, 300, 65), (8193, 192, 257, 24), (8064, 192, 256, 24),
                                     (8255, 63, 1024, 21), (3000, 784, 200, 196), (1023, 1024, 513, 128),
                                     (20_000, 320, 65, 64), (30_000, 16, 1025, 8), (23_000, 128, 129, 32),
                                     (20_000, 128, 128, 32), (3000, 64, 40, 16), (900, 10, 20, 2)])
@pytest.mark.parametrize("metric", ["l2", "ip"])
def test_lists_are_the_rule(n, d, L, M, metric):
    _check(_data(n, d, n + d + L), L, M, metric)


@pytest.mark.parametrize("kind", ["offset", "duplicates", "tiny", "huge", "bytes", "mixed"])
def test_hard_data(kind):
    import torch
    X = _data(40_001, 32, 5)
    if kind == "offset":  # every centroid inside the bound: 40,001 rows left to the FP32 tile kernel
        X = X + 300.0
    elif kind == "duplicates":  # equal centroids
        X = X[:200].repeat(201, 1)[:40_001].contiguous()
    elif kind in ("tiny", "huge"):
        X = X * (1e-9 if kind == "tiny" else 1e12)
    elif kind == "bytes":
        X = (128 + 20 * X).round().clamp(0, 255)
    else:
        X = X * torch.logspace(-6, 3, 32, device="cuda")
    _check(X, 300, 16, "l2", 2)


def test_more_rows_than_a_pass():
    _check(_data((1 << 20) + 133, 8, 9), 200, 4, "l2")
