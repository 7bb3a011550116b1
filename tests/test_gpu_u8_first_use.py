"""When the exact re-rank's U8 copies are made: not by the first searches of an
index, whose saving would not pay for them, but once a handle has re-ranked 16
candidates per row, and by a plan's creation (told by the device memory taken:
102 MB of copies); the results are those of the FP32 rows throughout."""
import pytest

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    g = torch.Generator(device="cuda").manual_seed(2)
    X = (20 * torch.randn((200_000, 512), generator=g, device="cuda") + 128).round().clamp(0, 255)
    Q = (20 * torch.randn((4096, 512), generator=g, device="cuda") + 128).clamp(0, 255)
    ix = ksc.build_index(X, 512, 64, iters=1)
    del X
    torch.cuda.empty_cache()
    return torch, ksc, ix, Q


def _taken(torch, f):
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    r = f()
    torch.cuda.synchronize()
    return r, before - torch.cuda.mem_get_info()[0]


def test_made_once_they_pay(env):
    torch, ksc, ix, Q = env
    v = ix.view()  # a handle of its own: nothing re-ranked yet
    ref = v.search(Q, 10, 4, 400, opts=ksc.search_opts(rerank_band=-1))  # warms the workspaces
    assert v.search(Q[:400], 10, 4, 400)[0].shape == (400, 10)
    total = 400 * 400
    made = False
    for _ in range(4):  # 1.6 M rows a search: 16 per row of the index is 3.2 M
        got, taken = _taken(torch, lambda: v.search(Q, 10, 4, 400))
        total += 4096 * 400
        assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
        assert (taken > 90 * MB) == (not made and total >= 16 * 200_000), (taken, total)
        made |= taken > 90 * MB
    assert made


def test_made_for_a_plan(env):
    torch, ksc, ix, Q = env
    v = ix.view()
    q = Q[:400].contiguous()
    ref = v.search(q, 10, 4, 100, opts=ksc.search_opts(rerank_band=-1))
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        plan, taken = _taken(torch, lambda: v.plan(400, 10, nprobe=4, rerank=100, stream=st))
        got = plan.execute(q, stream=st)
    st.synchronize()
    assert taken > 90 * MB
    assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
