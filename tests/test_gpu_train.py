"""The predictor's training (labels, sample order, minibatch gradients, Adam)
against the same run put together from public calls: labels from full searches
at every grid setting, gradients from ksc_mlp_grad, Adam in numpy.  Batches with
one and two partial-sum blocks, three (summed in no fixed order), and ragged
last ones.
"""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NPAR, K, TARGET, R_LAB = 8450, 10, 8, 100
GRID, RGRID = np.array([1, 2, 4, 8, 16], np.int32), np.array([12, 20, 40, 100], np.int32)


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    g = torch.Generator().manual_seed(3)
    X = torch.randn(6000, 32, generator=g)
    T = torch.randn(700, 32, generator=g) * 0.9
    ix = ksc.build_index(X.cuda(), 64, 16, seed=5)
    D = (T.double() ** 2).sum(1, keepdim=True) - 2 * T.double() @ X.double().T + (X.double() ** 2).sum(1)[None]
    kth = torch.topk(D, K, dim=1, largest=False).values[:, K - 1].float().cuda()
    return torch, ksc, ix, T.cuda(), kth


class SplitMix64:
    def __init__(self, s):
        self.s = s

    def __call__(self):
        mask = (1 << 64) - 1
        self.s = (self.s + 0x9E3779B97F4A7C15) & mask
        z = self.s
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        return z ^ (z >> 31)


def _labels(torch, ix, T, kth):
    tol = 1e-5 * kth.abs() + 1e-6

    def found(dists):
        return (dists <= (kth + tol)[:, None]).sum(1) >= TARGET

    n = torch.full((len(T),), int(GRID[-1]), dtype=torch.int32, device="cuda")
    for p in GRID[::-1]:
        n[found(ix.search(T, K, int(p), R_LAB)[1])] = int(p)
    r = torch.full_like(n, int(RGRID[-1]))
    for v in RGRID[::-1]:
        _, dists = ix.search_varprobe(T, K, n, torch.full_like(n, int(v)), nprobe_max=int(GRID[-1]))
        r[found(dists)] = int(v)
    # a later grid value may miss what an earlier one found: the smallest counts,
    # which the descending order above keeps
    return n.cpu().numpy(), r.cpu().numpy()


@pytest.mark.parametrize("batch", [64, 100, 256, 300])
def test_training_equals_its_parts(env, batch):
    torch, ksc, ix, T, kth = env
    lr, seed, epochs, nt = 1e-3, 11, 2, len(T)
    loss = ix.train_predictor(T, kth, k=K, target_hits=TARGET, rerank_label=R_LAB, epochs=epochs, batch=batch, lr=lr,
                              seed=seed, grid=GRID, rgrid=RGRID)
    got = ix.predictor_weights()
    ln, lrk = _labels(torch, ix, T, kth)
    assert len(np.unique(ln)) > 2
    Y = np.stack([l > np.sort(l)[nt // 2] for l in (ln, lrk)], 1).astype(np.float32)
    feats = ix.query_features(T)
    rnd = SplitMix64(seed)
    w = np.zeros(NPAR, np.float32)
    off = 0
    for rows in (64, 64, 2):
        a = np.float32(np.sqrt(np.float32(6) / np.float32(64)))
        for e in range(rows * 64):
            w[off + e] = a * (np.float32(2) * np.float32((rnd() >> 11) * 2.0 ** -53) - np.float32(1))
        off += rows * 64 + rows
    m, v = np.zeros_like(w), np.zeros_like(w)
    f = np.float32
    g, ls = torch.empty(NPAR, device="cuda"), torch.empty(1, device="cuda")
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    t = 0
    for _ in range(epochs):
        perm = np.arange(nt)
        for i in range(nt - 1, 0, -1):
            j = rnd() % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        losses = []
        for b in range(0, nt, batch):
            sel = perm[b:b + batch]
            x = feats[torch.from_numpy(sel).cuda()].contiguous()
            y = torch.from_numpy(Y[sel]).cuda()
            wd = torch.from_numpy(w).cuda()
            assert ksc.lib().ksc_mlp_grad(*(C.c_void_p(z.data_ptr()) for z in (wd, x, y)), len(sel),
                                          *(C.c_void_p(z.data_ptr()) for z in (g, ls)), st) == 0
            gi = g.cpu().numpy()
            losses.append(ls.item())
            t += 1
            m = f(0.9) * m + (f(1) - f(0.9)) * gi
            v = f(0.999) * v + (f(1) - f(0.999)) * gi * gi
            w = w - f(lr) * (m / f(1 - f(0.9) ** f(t))) / (np.sqrt(v / f(1 - f(0.999) ** f(t))) + f(1e-8))
    # a step is at most a few lr; roundings are 2^-24 relative per operation,
    # amplified only where a gradient is a small difference of large terms.  A wrong
    # sample, label or order moves most weights by the order of lr.
    err = np.abs(got - w) / (lr * t)
    assert abs(loss - np.mean(losses)) <= 1e-4 * np.mean(losses)
    assert np.median(err) <= 1e-3 and np.quantile(err, 0.99) <= 2e-2
