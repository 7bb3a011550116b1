"""Training steps of more samples than the spread kernels take (gathered, a CTA
per 128 samples), up to a batch far above the samples there are (whose scratch
is that of the samples): the predictor against the run put together from its
parts, the pruner against nearly the same minibatches on the spread kernels."""
import numpy as np
import pytest

import test_gpu_train as parts

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    g = torch.Generator().manual_seed(3)
    X = torch.randn(6000, 32, generator=g)
    T = torch.randn(8700, 32, generator=g) * 0.9
    ix = ksc.build_index(X.cuda(), 64, 16, seed=5)
    kth = torch.cat([torch.topk((t * t).sum(1, keepdim=True) - 2 * t @ X.double().T + (X.double() ** 2).sum(1)[None],
                                parts.K, dim=1, largest=False).values[:, -1] for t in T.double().split(1000)])
    return torch, ksc, ix, T.cuda(), kth.float().cuda()


@pytest.mark.parametrize("batch", [8192, 8193, 1 << 28])
def test_predictor_equals_its_parts(env, batch):
    parts.test_training_equals_its_parts(env, batch)


def test_pruner_beside_the_spread_steps(env):
    torch, ksc, ix, T, kth = env
    ix.pruner_stats(iters=4)
    got = []
    for batch in (2048, 2049, 1 << 28):  # 4096 rows: 2048 + 2048, 2049 + 2047, all
        loss = ix.train_pruner(T[:256].contiguous(), kth[:256].contiguous(), P=16, epochs=1, batch=batch, lr=1e-3, seed=7)
        assert np.isfinite(loss)
        got.append(ix.pruner_model())
    d = np.abs(got[0] - got[1]) / 2e-3  # of two steps of at most about lr
    # a sample in 2048 moves a gradient by about its own share, and Adam's steps
    # where that is small against the gradient by as little; other samples, sums or
    # moments move most weights by the order of a step
    assert np.median(d) <= 1e-2 and np.quantile(d, 0.9) <= 0.2
    assert np.isfinite(got[2]).all()
