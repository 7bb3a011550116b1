"""Performance cases of the KScaNN library: what a program that uses it has it do.

A case fixes an index (its data, sizes, metric), a batch of queries and the
search settings; `run` makes one pass through the public entry points.  The
indexes are made here in torch from the seed (centroids by two Lloyd rounds on
a sample, codebooks by k-means on residuals) and imported, as a program does
that loads an index it built before; the build and training cases start from
the raw vectors and queries.

Real-valued data are rounded to FP16 values, as stored embeddings are, so the
FP64 sums behind every centroid are exact in any order and two preparations of
one seed are equal bit for bit.
"""
import math

import numpy as np
import torch

from paper_2511_03298_gb300 import ksc

DEV = "cuda"


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # batch-1 serving: one SIFT-shaped query at a time, replayed from a captured plan
        dict(name="one_query_plan", kind="search", data="bytes", metric="l2", n=1_000_000, d=128, L=1024, M=64,
             nq=1, k=10, nprobe=7, R=200, plan=True, precision=0, Rf=0),
        # a small collection and a small batch through the direct call (the 10k x 128 configuration)
        dict(name="small_100", kind="search", data="mixture", metric="l2", n=10_000, d=128, L=64, M=64, nq=100, k=10,
             nprobe=8, R=100, plan=False, precision=0, Rf=0),
        # a handful of queries that probe widely and want many neighbours (DEEP shape)
        dict(name="deep_16", kind="varprobe", data="unit", metric="l2", n=1_000_000, d=96, L=4096, M=48, nq=16,
             k=100, pmin=4, pmax=256, rmin=500, R=1000),
        # the same at an ordinary server batch, nprobe and rerank different for every query
        dict(name="deep_1024", kind="varprobe", data="unit", metric="l2", n=2_000_000, d=96, L=4096, M=48, nq=1024,
             k=100, pmin=4, pmax=256, rmin=500, R=1000),
        # the throughput configuration: 10k SIFT-shaped queries against 1M vectors, fixed nprobe
        dict(name="sift_10k", kind="search", data="bytes", metric="l2", n=1_000_000, d=128, L=1024, M=64, nq=10_000,
             k=10, nprobe=8, R=200, plan=False, precision=0, Rf=0),
        # the same with nprobe and rerank predicted per query, replayed from a captured plan
        dict(name="adaptive_10k", kind="adaptive", data="bytes", metric="l2", n=1_000_000, d=128, L=1024, M=64,
             nq=10_000, k=10, pmin=4, pmax=12, rmin=80, R=200, plan=True),
        # maximum inner product on embeddings (GLOVE shape, M not a multiple of the lanes)
        dict(name="inner_product_10k", kind="search", data="unit", metric="ip", n=600_000, d=100, L=1024, M=50,
             nq=10_000, k=10, nprobe=16, R=200, plan=False, precision=0, Rf=0),
        # the same through the widened BF16 shortlist, an odd batch
        dict(name="shortlist_bf16", kind="search", data="unit", metric="ip", n=600_000, d=100, L=1024, M=50, nq=3001,
             k=10, nprobe=16, R=400, plan=False, precision=1, Rf=100),
        # long vectors: 28 x 28 images, exact re-rank over 784 dimensions
        dict(name="images_784", kind="search", data="image", metric="l2", n=60_000, d=784, L=256, M=196, nq=10_000,
             k=10, nprobe=4, R=200, plan=False, precision=0, Rf=0),
        # the hybrid leaf search: near lists scanned, the graphs of the others walked
        dict(name="hybrid_2000", kind="hybrid", data="mixture", metric="l2", n=100_000, d=64, L=128, M=32, nq=2000,
             k=10, nprobe=12, R=100, near=2, efs=64, tau=8),
        # indexing: k-means, codebooks, encoding and packing of new vectors
        dict(name="build_200k", kind="build", data="bytes", metric="l2", n=200_000, d=128, L=512, M=64, iters=20,
             graph=False),
        # training the nprobe / rerank predictor on labelled queries
        dict(name="train_16k", kind="train", data="bytes", metric="l2", n=100_000, d=128, L=256, M=64, nq=16_384,
             k=10, epochs=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "search", "varprobe", "adaptive", "hybrid", "build", "train"])
    if kind == "build":
        d, M = rng.choice([(128, 64), (128, 32), (96, 48), (100, 50), (64, 16)])
        n = _log(rng, 10_000, 200_000)
        return dict(kind=kind, data=rng.choice(["bytes", "unit"]), metric=rng.choice(["l2", "l2", "ip"]), n=n, d=d,
                    L=_log(rng, 32, min(512, n // 100)), M=M, iters=rng.choice([10, 20]),
                    graph=n <= 60_000 and rng.random() < 0.5)
    if kind == "train":
        return dict(kind=kind, data="bytes", metric="l2", n=_log(rng, 20_000, 100_000), d=128, L=_log(rng, 96, 256),
                    M=rng.choice([32, 64]), nq=_log(rng, 2000, 12_000), k=10, epochs=rng.choice([4, 8]))
    if kind == "hybrid":
        d, M = rng.choice([(64, 32), (32, 16), (128, 64)])
        n = _log(rng, 20_000, 100_000)
        return dict(kind=kind, data="mixture", metric="l2", n=n, d=d, L=max(24, n // 800), M=M, nq=_log(rng, 10, 2000),
                    k=10, nprobe=rng.randint(4, 12), R=rng.choice([60, 100, 200]), near=rng.choice([1, 2, 3]),
                    efs=rng.choice([32, 64]), tau=rng.choice([4, 8]))
    if kind == "varprobe":
        return dict(kind=kind, data="unit", metric="l2", n=_log(rng, 100_000, 1_000_000), d=96, L=_log(rng, 512, 4096),
                    M=48, nq=_log(rng, 4, 1024), k=rng.choice([10, 50, 100]), pmin=4, pmax=rng.randint(32, 256),
                    rmin=200, R=rng.choice([400, 1000]))
    if kind == "adaptive":
        return dict(kind=kind, data="bytes", metric="l2", n=_log(rng, 100_000, 1_000_000), d=128,
                    L=_log(rng, 256, 1024), M=rng.choice([32, 64]), nq=_log(rng, 16, 10_000), k=10, pmin=4,
                    pmax=rng.randint(8, 24), rmin=rng.choice([50, 80]), R=200, plan=rng.random() < 0.5)
    data = rng.choice(["bytes", "mixture", "unit", "unit", "image"])
    metric = "l2" if data in ("bytes", "image") else rng.choice(["l2", "ip"])
    if data == "image":
        d, M, n = 784, 196, _log(rng, 20_000, 60_000)
    else:
        d, M = rng.choice([(128, 64), (128, 32), (96, 48), (100, 50), (64, 32), (64, 16)])
        n = _log(rng, 10_000, 1_000_000)
    L = max(32, min(1024, int(math.sqrt(n) * rng.uniform(0.5, 1.0))))
    k = rng.choice([1, 10, 10, 20, 50])
    precision = rng.choice([0, 0, 0, 1, 2])
    R = rng.choice([100, 200, 333, 400])
    return dict(kind=kind, data=data, metric=metric, n=n, d=d, L=L, M=M, nq=_log(rng, 1, 10_000), k=k,
                nprobe=rng.randint(2, 12), R=R, plan=rng.random() < 0.3, precision=precision,
                Rf=100 if precision else 0)


# ------------------------------------------------------------------ inputs, on the GPU, from the seed
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _normal(shape, g):
    return torch.randn(shape, generator=g, device=DEV)


def _uniform(shape, g):
    return torch.rand(shape, generator=g, device=DEV)


def _f16(x):
    return x.half().float()


def _mixture(case, seed):
    """The mixture of a seed: draw(m, g) gives m vectors of it."""
    g, d, data = _gen(seed), case["d"], case["data"]
    if data == "bytes":  # SIFT shape: crowded components on skewed scales, integers 0..255
        s = torch.exp(0.5 * _normal((d,), g))
        sup = _uniform((30, d), g) * (96.0 * s)
        mu = sup[torch.randint(0, 30, (1000,), generator=g, device=DEV)] + _normal((1000, d), g) * (10.0 * s)

        def make(m, h):
            c = torch.randint(0, 1000, (m,), generator=h, device=DEV)
            return (mu[c] + 20.0 * s * _normal((m, d), h)).round_().clamp_(0, 255)
    elif data == "mixture":  # 100 Gaussian clusters, real-valued
        mu = _uniform((100, d), g) * 10.0 - 5.0

        def make(m, h):
            c = torch.randint(0, 100, (m,), generator=h, device=DEV)
            return _f16(mu[c] + _normal((m, d), h))
    elif data == "unit":  # embeddings of unit norm, components of very different weight
        nc = 2000
        mu = torch.nn.functional.normalize(_normal((nc, d), g), dim=1)
        sig = 0.06 * torch.exp(0.4 * _normal((nc, d), g))
        cw = torch.cumsum(1.0 / torch.arange(1, nc + 1, dtype=torch.float64, device=DEV) ** 0.6, 0)

        def make(m, h):
            u = torch.rand((m,), generator=h, device=DEV, dtype=torch.float64) * cw[-1]
            c = torch.searchsorted(cw, u).clamp_(max=nc - 1)
            return _f16(torch.nn.functional.normalize(mu[c] + sig[c] * _normal((m, d), h), dim=1))
    else:  # image: smooth 28 x 28 templates with pixel noise and an almost empty border
        px = torch.arange(28, device=DEV).float()
        tpl = torch.zeros((100, 28, 28), device=DEV)
        for _ in range(4):
            cy, cx = 5.0 + 17.0 * _uniform((100, 1, 1), g), 5.0 + 17.0 * _uniform((100, 1, 1), g)
            sy, sx = 2.0 + 4.0 * _uniform((100, 1, 1), g), 2.0 + 4.0 * _uniform((100, 1, 1), g)
            tpl += (100.0 + 155.0 * _uniform((100, 1, 1), g)) * torch.exp(
                -0.5 * (((px[:, None] - cy) / sy) ** 2 + ((px[None, :] - cx) / sx) ** 2))
        inner = torch.zeros((28, 28), device=DEV)
        inner[2:26, 2:26] = 1.0
        mu, inner = (tpl.clamp_(0, 255) * inner).reshape(100, -1), inner.reshape(-1)

        def make(m, h):
            c = torch.randint(0, 100, (m,), generator=h, device=DEV)
            x = mu[c] * (0.7 + 0.6 * _uniform((m, 1), h)) + 25.0 * _normal((m, 784), h)
            return x.round_().clamp_(0, 255).mul_(inner)
    return make


def _vectors(case, seed, m, stream):
    make, g = _mixture(case, seed), _gen(seed * 7 + stream)
    return torch.cat([make(min(1 << 18, m - b), g) for b in range(0, m, 1 << 18)])


def _nearest(X, C, spherical):
    """Nearest centroid of every row (ties to the lower id), in FP32 on the GPU."""
    base = 0.0 if spherical else C.square().sum(1)
    out = torch.empty(X.shape[0], dtype=torch.int64, device=DEV)
    step = max(1, (1 << 28) // C.shape[0])
    for b in range(0, X.shape[0], step):
        s = X[b:b + step] @ C.t()
        out[b:b + step] = (base - (1.0 if spherical else 2.0) * s).argmin(1)
    return out


def _means(X, a, C):
    """Mean of every centroid's rows in FP64 (an empty one keeps its centroid)."""
    L, d = C.shape
    s = torch.zeros((L, d), dtype=torch.float64, device=DEV)
    for b in range(0, X.shape[0], 1 << 18):
        s.index_add_(0, a[b:b + (1 << 18)], X[b:b + (1 << 18)].double())
    cnt = torch.bincount(a, minlength=L).double()[:, None]
    return torch.where(cnt > 0, s / cnt.clamp(min=1), C.double()).float()


def _codes(R, cb):
    """Nearest codeword of every (row, subspace); R [m x M x dsub], cb [M x 16 x dsub]."""
    out = torch.empty(R.shape[:2], dtype=torch.uint8, device=DEV)
    step = max(1, (1 << 27) // R.shape[1] // 16)
    for b in range(0, R.shape[0], step):
        acc = 0.0
        for t in range(R.shape[2]):
            acc = acc + (R[b:b + step, :, None, t] - cb[None, :, :, t]).square()
        out[b:b + step] = acc.argmin(2).to(torch.uint8)
    return out


def _arrays(case, seed):
    """The index of a case: vectors, centroids, lists, codebooks, codes (GPU tensors)."""
    n, d, L, M = case["n"], case["d"], case["L"], case["M"]
    spherical = case["metric"] == "ip"
    X = _vectors(case, seed, n, 1)
    pick = torch.randperm(n, generator=_gen(seed + 5), device=DEV)
    C, sample = X[pick[:L]], X[pick[:min(n, 32 * L)]]
    for _ in range(2):
        C = _means(sample, _nearest(sample, C, False), C)
    c_rank = torch.nn.functional.normalize(C.double(), dim=1).float() if spherical else C
    assign = _nearest(X, c_rank, spherical)
    c_mean = _means(X, assign, C)
    rs = pick[:min(n, 8192)]
    S = (X[rs] - c_mean[assign[rs]]).view(-1, M, d // M)
    cb = S[:16].transpose(0, 1).contiguous()
    for _ in range(4):
        hot = torch.nn.functional.one_hot(_codes(S, cb).long(), 16).permute(1, 2, 0).double()  # M x 16 x rows
        cnt = hot.sum(2, keepdim=True)
        cb = torch.where(cnt > 0, torch.bmm(hot, S.transpose(0, 1).double()) / cnt.clamp(min=1), cb.double()).float()
    codes = torch.empty((n, M), dtype=torch.uint8, device=DEV)
    for b in range(0, n, 1 << 18):
        a = assign[b:b + (1 << 18)]
        codes[b:b + (1 << 18)] = _codes((X[b:b + (1 << 18)] - c_mean[a]).view(-1, M, d // M), cb)
    return dict(X=X, c_rank=c_rank, c_mean=c_mean, codebook=cb, codes=codes, assign=assign.int())


def _graph(A, L):
    """32 nearest members of its own list for every vector, and each list's entry."""
    X, a = A["X"], A["assign"].long()
    graph = torch.full((X.shape[0], 32), -1, dtype=torch.int32, device=DEV)
    entry = torch.full((L,), -1, dtype=torch.int32, device=DEV)
    for p in range(L):
        m = (a == p).nonzero()[:, 0]
        if len(m) == 0:
            continue
        x = X[m]
        entry[p] = m[(x - A["c_mean"][p]).square().sum(1).argmin()]
        kk = min(32, len(m) - 1)
        if kk > 0:
            sq = x.square().sum(1)
            D = (sq[:, None] + sq[None, :] - 2.0 * (x @ x.t())).fill_diagonal_(math.inf)
            graph[m, :kk] = m[D.topk(kk, 1, largest=False).indices].int()
    return graph, entry


def _host(A):
    return {key: v.cpu().numpy() for key, v in A.items()}


def _predictor(seed):
    """Predictor weights of a seed (He-uniform layers, a wide output layer), packed as the library packs them."""
    r = np.random.default_rng(seed)
    parts = []
    for rows, fan, gain in ((64, 64, 1.0), (64, 64, 1.0), (2, 64, 0.5)):
        parts += [gain * math.sqrt(6.0 / fan) * r.uniform(-1, 1, rows * fan), np.zeros(rows)]
    return np.concatenate(parts).astype(np.float32)


def _settings(case, seed):
    """Per-query nprobe and rerank of a varprobe case."""
    g = _gen(seed + 11)
    P = torch.randint(case["pmin"], case["pmax"] + 1, (case["nq"],), generator=g, device=DEV, dtype=torch.int32)
    R = torch.randint(case["rmin"], case["R"] + 1, (case["nq"],), generator=g, device=DEV, dtype=torch.int32)
    return P, R


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "build":
        s["X"] = _vectors(case, seed, case["n"], 1)
        return s
    A = _arrays(case, seed)
    s["Q"] = _vectors(case, seed, case["nq"], 2)
    if kind == "hybrid":
        A["graph"], A["entry"] = _graph(A, case["L"])
    if kind == "train":  # the true k-th distances (integer vectors: exact in FP32)
        xx, kth = A["X"].square().sum(1), []
        for b in range(0, case["nq"], 2048):
            q = s["Q"][b:b + 2048]
            D = q.square().sum(1, keepdim=True) + xx - 2.0 * (q @ A["X"].t())
            kth.append(D.kthvalue(case["k"], 1).values if D.shape[1] < 2048 else
                       D.topk(case["k"], 1, largest=False).values[:, -1])
        s["kth"] = torch.cat(kth).contiguous()
    s["ix"] = ksc.index_import(_host(A), metric=case["metric"])
    if kind == "varprobe":
        s["P"], s["R"] = _settings(case, seed)
    if kind == "adaptive":
        s["ix"].predictor_weights(_predictor(seed))
        s["ix"].set_predictor_params(case["pmin"], case["pmax"], case["rmin"], case["R"], 0.3, 0.5, 0.3, 0.5)
    s["opts"] = None
    if kind == "hybrid":
        s["opts"] = ksc.search_opts(hybrid=True, n_near=case["near"], efs=case["efs"], tau=case["tau"])
    if case.get("precision"):
        s["opts"] = ksc.search_opts(precision=case["precision"], rerank_final=case["Rf"])
    if case.get("plan"):
        s["stream"] = torch.cuda.Stream()
        s["stream"].wait_stream(torch.cuda.current_stream())
        s["plan"] = s["ix"].plan(case["nq"], case["k"], nprobe=case.get("nprobe", 1), rerank=case["R"],
                                 adaptive=kind == "adaptive", opts=s["opts"], stream=s["stream"])
        s["out"] = (torch.empty((case["nq"], case["k"]), dtype=torch.int64, device=DEV),
                    torch.empty((case["nq"], case["k"]), device=DEV))
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "build":
        ix = ksc.build_index(s["X"], c["L"], c["M"], metric=c["metric"], iters=c["iters"], build_graph=c["graph"])
        e = ix.export(with_graph=c["graph"], fields=("c_rank", "c_mean", "codebook", "codes", "assign"))
        return [v for v in e.values() if isinstance(v, np.ndarray)]
    if kind == "train":
        loss = s["ix"].train_predictor(s["Q"], s["kth"], k=c["k"], epochs=c["epochs"])
        return [s["ix"].predictor_weights(), loss]
    if c.get("plan"):  # plans are captured and replayed on a stream of their own
        here = torch.cuda.current_stream()
        s["stream"].wait_stream(here)
        out = s["plan"].execute(s["Q"], *s["out"], stream=s["stream"])
        here.wait_stream(s["stream"])
        return list(out)
    if kind == "varprobe":
        return list(s["ix"].search_varprobe(s["Q"], c["k"], s["P"], s["R"], c["pmax"], c["R"]))
    if kind == "adaptive":
        return list(s["ix"].search_adaptive(s["Q"], c["k"]))
    return list(s["ix"].search(s["Q"], c["k"], c["nprobe"], c["R"], opts=s["opts"]))


# ------------------------------------------------------------------ the work a pass cannot do without
def work(c):
    n, d, L, M = c["n"], c["d"], c["L"], c["M"]
    if c["kind"] == "build":
        ns, npq = min(n, 256 * L), min(n, 65536)
        graph = n * (n / L) * d * 3 if c["graph"] else 0
        flops = 2.0 * d * L * (ns * c["iters"] + n) + 3.0 * 16 * d * (npq * c["iters"] + n) + graph
        return dict(bytes=4.0 * n * d + n * M + 4.0 * n + 8.0 * L * d + 64.0 * d + (132.0 * n if c["graph"] else 0),
                    flops=flops)
    nq = c["nq"]
    if c["kind"] == "train":  # labels: the default grids' scans and re-ranks; then the epochs
        P, R, out = sum(p for p in (4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128) if p <= L), 11 * 200 + 770, 4.0 * 8450
        extra = 6.0 * 8450 * nq * c["epochs"]
    else:
        P = c["nprobe"] if "nprobe" in c else 0.5 * (c["pmin"] + c["pmax"])
        R, out, extra = 0.5 * (c.get("rmin", c["R"]) + c["R"]), 12.0 * nq * c["k"], 0.0
    lists = min(1.0, nq * P / L)  # share of the lists that some query probes
    rows = min(float(n), nq * R)
    return dict(bytes=4.0 * nq * d + 4.0 * L * d + 64.0 * d + lists * (0.5 * n * M + 4.0 * L * d) + 4.0 * rows * d + out,
                flops=2.0 * nq * L * d + nq * P * (48.0 * d + n / L * M) + 3.0 * nq * R * d + extra)


# ------------------------------------------------------------------ the same in 64 bits
def _lut(A, Q, probes, P, ip):
    """8-bit tables [nq x Pmax x M x 16] and integer biases [nq x Pmax] by the LUT rule."""
    nq, Pm = probes.shape
    M, _, ds = A["codebook"].shape
    cb, cm = A["codebook"].double(), A["c_mean"].double()
    live = torch.arange(Pm, device=DEV)[None] < P[:, None]
    lut = torch.empty((nq, Pm, M, 16), dtype=torch.uint8, device=DEV)
    bias = torch.empty((nq, Pm), dtype=torch.int64, device=DEV)
    step = max(1, (1 << 27) // (Pm * M * 16))
    for b in range(0, nq, step):
        q, pr = Q[b:b + step].double(), probes[b:b + step]
        u = (q[:, None].expand(-1, Pm, -1) if ip else q[:, None] - cm[pr]).reshape(len(q), Pm, M, ds)
        T = 0.0
        for t in range(ds):
            w = cb[None, None, :, :, t]
            T = T - u[..., t, None] * w if ip else T + (u[..., t, None] - w).square()
        lo = T.amin(3)
        span = torch.where(live[b:b + step], (T.amax(3) - lo).amax(2), 0.0).amax(1)
        a = torch.where(span == 0, 1.0, 255.0 / span)
        S = lo.sum(2) - ((q[:, None] * cm[pr]).sum(2) if ip else 0.0)
        lut[b:b + step] = torch.floor((T - lo[..., None]) * a[:, None, None, None] + 0.5).clamp(0, 255).to(torch.uint8)
        bias[b:b + step] = torch.floor(S * a[:, None] + 0.5).long()
    return lut, bias


def _candidates(A, probes, P, lut, bias, Rmax):
    """Keys D 2^32 + id of the Rmax best vectors of every query's lists."""
    nq, Pm = probes.shape
    L, M = A["c_rank"].shape[0], A["codes"].shape[1]
    assign = A["assign"].long()
    size = torch.bincount(assign, minlength=L)
    order = torch.sort(assign, stable=True).indices
    first = torch.cumsum(size, 0) - size
    live = torch.arange(Pm, device=DEV)[None] < P[:, None]
    take = torch.where(live, size[probes], 0)
    off = torch.cumsum(take, 1) - take
    W = max(int(take.sum(1).max()), Rmax)
    keys = torch.full((nq * W,), torch.iinfo(torch.int64).max, device=DEV)
    pair = live.reshape(-1).nonzero()[:, 0]
    pair = pair[torch.sort(probes.reshape(-1)[pair], stable=True).indices]
    per = torch.bincount(probes.reshape(-1)[pair], minlength=L).tolist()
    lut2, at = lut.view(nq * Pm, M * 16), 0
    sizes, firsts = size.tolist(), first.tolist()
    cols = 16 * torch.arange(M, device=DEV)
    for p in range(L):
        if not per[p] or not sizes[p]:
            at += per[p]
            continue
        e, ids = pair[at:at + per[p]], order[firsts[p]:firsts[p] + sizes[p]]
        at += per[p]
        hot = torch.zeros((len(ids), M * 16), device=DEV).scatter_(1, cols + A["codes"][ids].long(), 1.0)
        D = (lut2[e].float() @ hot.t()).long() + bias.reshape(-1)[e][:, None]  # integers below 2^24: exact
        pos = (e // Pm * W + off.reshape(-1)[e])[:, None] + torch.arange(len(ids), device=DEV)
        keys[pos.reshape(-1)] = ((D << 32) + ids).reshape(-1)
    return keys.view(nq, W).topk(Rmax, 1, largest=False, sorted=True).values


def _rows(X, Q, ids, ok, ip):
    """FP64 distances (or negated similarities) of every query to its candidate rows."""
    out = torch.empty(ids.shape, dtype=torch.float64, device=DEV)
    step = max(1, (1 << 26) // (ids.shape[1] * X.shape[1]))
    for b in range(0, len(Q), step):
        x, q = X[ids[b:b + step]].double(), Q[b:b + step, None].double()
        out[b:b + step] = -(x * q).sum(2) if ip else (x - q).square().sum(2)
    return torch.where(ok, out, math.inf)


def exact(case, seed):
    """Distances of a search in FP64 (ids are whole numbers; a walk of the graphs,
    k-means and training have no value that does not hang on their own choices)."""
    kind = case["kind"]
    if kind in ("build", "train", "hybrid") or case.get("precision") == 2:
        return None
    A, Q, k, L = _arrays(case, seed), _vectors(case, seed, case["nq"], 2), case["k"], case["L"]
    ip, nq, Rmax = case["metric"] == "ip", case["nq"], max(case["R"], case["k"])
    C = A["c_rank"].double()
    score = -(Q.double() @ C.t()) if ip else C.square().sum(1) - 2.0 * (Q.double() @ C.t())
    if kind == "varprobe":
        P, R = (t.long() for t in _settings(case, seed))
        R = R.clamp(min=k)
    elif kind == "adaptive":
        f = score.topk(32, 1, largest=False, sorted=True).values + (1.0 if ip else Q.double().square().sum(1)[:, None])
        f = f.clamp(min=0)
        bf = lambda v: v.float().bfloat16().double()  # noqa: E731
        h = bf(torch.cat([(f + 1e-12) / (f.mean(1, keepdim=True) + 1e-12), (f[:, :1] + 1e-12) / (f + 1e-12)], 1))
        w, at = torch.from_numpy(_predictor(seed)).to(DEV), 0
        for rows in (64, 64, 2):
            W, b = w[at:at + rows * 64].view(rows, 64), w[at + rows * 64:at + rows * 65]
            h, at = h @ bf(W).t() + bf(b), at + rows * 65
            h = bf(h.relu()) if rows == 64 else torch.sigmoid(h)

        def eq2(p, lo, hi):
            return (lo + torch.ceil((hi - lo) * (p - 0.3).clamp(min=0) * (p + 0.5))).clamp(max=hi).long()
        P, R = eq2(h[:, 0], case["pmin"], case["pmax"]), eq2(h[:, 1], case["rmin"], case["R"]).clamp(min=k)
    else:
        P, R = (torch.full((nq,), v, device=DEV) for v in (case["nprobe"], Rmax))
    probes = score.topk(min(int(P.max()), L), 1, largest=False, sorted=True).indices
    del score
    lut, bias = _lut(A, Q, probes, P, ip)
    keys = _candidates(A, probes, P, lut, bias, Rmax)
    del lut
    ids = keys & 0xffffffff
    ok = (keys != torch.iinfo(torch.int64).max) & (torch.arange(Rmax, device=DEV)[None] < R[:, None])
    ids = torch.where(ok, ids, 0)
    if case.get("precision") == 1:  # the shortlist by BF16 rows first
        D = _rows(A["X"].bfloat16(), Q, ids, ok, ip)
        best = D.topk(max(case["Rf"], k), 1, largest=False, sorted=True).indices
        ids, ok = ids.gather(1, best), ok.gather(1, best)
    D = _rows(A["X"], Q, ids, ok, ip)
    D = D.sort(1).values[:, :k]
    out = [None, -D if ip else D]
    if kind == "adaptive" and not case["plan"]:
        out += [None, None]
    return out
