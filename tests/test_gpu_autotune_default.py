"""The autotuner times the scan that the batch takes by itself beside the lanes it
can ask for: where many queries share the lists that is the tensor-core scan, a
third faster than any lanes at this size, and the tuned options leave it on.
Where the batch takes byte permutes anyway, or the caller asks for the
tensor-core scan, lanes are returned as before.  The tuned options follow the
rule on other batches too."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    g = torch.Generator(device="cuda").manual_seed(4)
    mu = torch.randn(500, 128, generator=g, device="cuda")
    X = mu[torch.randint(0, 500, (200_000,), generator=g, device="cuda")] + 0.5 * torch.randn(200_000, 128, generator=g, device="cuda")
    Q = mu[torch.randint(0, 500, (4000,), generator=g, device="cuda")] + 0.5 * torch.randn(4000, 128, generator=g, device="cuda")
    return ksc, ksc.build_index(X, 256, 64, iters=3), Q


def test_shared_lists_keep_the_tensor_core_scan(env):
    import torch
    ksc, ix, Q = env
    opts, ms = ix.autotune(Q, 10, 8, 200)
    assert opts.scan_tc == 2 and opts.lanes_per_query in (4, 8, 16, 32)
    assert opts.tile_blocks in (0, 8, 16, 32, 64) and ms > 0
    for nq in (4000, 300, 3):
        q = Q[:nq].contiguous()
        a, b = ix.search(q, 10, 8, 200), ix.search(q, 10, 8, 200, opts=opts)
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


@pytest.mark.parametrize("nq,ask", [(1000, False), (500, True), (4000, True), (20, False)])
def test_lanes_elsewhere(env, nq, ask):
    import torch
    ksc, ix, Q = env
    q, P = Q[:nq].contiguous(), 3 if not ask else 8
    if not ask:
        assert nq * P < 20 * 256
    opts, _ = ix.autotune(q, 10, P, 100, opts=ksc.search_opts(scan_tc=ask))
    assert opts.scan_tc == int(ask) and opts.lanes_per_query in (4, 8, 16, 32)
    a, b = ix.search(q, 10, P, 100), ix.search(q, 10, P, 100, opts=opts)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


def test_tuned_options_tuned_again(env):
    ksc, ix, Q = env
    opts, _ = ix.autotune(Q, 10, 8, 200)
    again, _ = ix.autotune(Q[:1000].contiguous(), 10, 3, 100, opts=opts)  # a batch that takes byte permutes
    assert again.scan_tc == 0 and again.lanes_per_query in (4, 8, 16, 32)


def test_bad_arguments_are_refused(env):
    ksc, ix, Q = env
    for k, P, R in ((0, 8, 200), (10, 0, 200), (10, 257, 200), (10, 8, 5000)):
        with pytest.raises(Exception):
            ix.autotune(Q[:100].contiguous(), k, P, R)
