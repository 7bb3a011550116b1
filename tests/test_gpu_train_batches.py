"""A training batch far above the samples there are: the scratch is that of the
samples, and the run equals the one put together from its parts."""
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


@pytest.mark.parametrize("batch", [1 << 28])
def test_predictor_equals_its_parts(env, batch):
    parts.test_training_equals_its_parts(env, batch)
