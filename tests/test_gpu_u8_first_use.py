"""When the exact re-rank's U8 copies are made: not by the first searches of an
index, whose saving would not pay for them, but once a handle has re-ranked 16
candidates per row, by a plan's creation and when the band is asked for (told by the device memory taken:
102 MB of copies); the results are those of the FP32 rows throughout.  Where the
device has no room for them the search goes on without, and they are made later."""
import ctypes as C

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


@pytest.mark.parametrize("nq,R", [(400, 51), (304, 200)])
def test_made_when_asked_for(env, nq, R):
    torch, ksc, ix, Q = env
    v = ix.view()
    q = Q[:nq].contiguous()
    ref = v.search(q, 10, 4, R, opts=ksc.search_opts(rerank_band=-1))
    v.search(q, 10, 4, R)
    got, taken = _taken(torch, lambda: v.search(q, 10, 4, R, opts=ksc.search_opts(rerank_band=1)))
    assert taken > 90 * MB
    assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])


def test_made_later_where_there_was_no_room(env):
    torch, ksc, ix, Q = env
    v = ix.view()
    ref = v.search(Q, 10, 4, 400, opts=ksc.search_opts(rerank_band=-1))
    v.search(Q, 10, 4, 400)
    rt = C.CDLL("libcudart.so.13")
    rt.cudaMalloc.argtypes, rt.cudaFree.argtypes = [C.POINTER(C.c_void_p), C.c_size_t], [C.c_void_p]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    out = torch.empty((4096, 10), dtype=torch.int64, device="cuda"), torch.empty((4096, 10), device="cuda")
    held = []
    try:
        for size in (8 << 30, 512 * MB, 16 * MB):
            while torch.cuda.mem_get_info()[0] >= 60 * MB + size:
                p = C.c_void_p()
                if rt.cudaMalloc(C.byref(p), size):
                    break
                held.append(p)
        for _ in range(2):  # the copies are due, and 102 MB are not to be had
            v.search(Q, 10, 4, 400, out=out)
            torch.cuda.synchronize()
    finally:
        for p in held:
            assert rt.cudaFree(p) == 0
    assert torch.equal(out[0], ref[0]) and torch.equal(out[1], ref[1])
    made = 0
    for _ in range(3):
        got, taken = _taken(torch, lambda: v.search(Q, 10, 4, 400))
        made += taken > 90 * MB
        assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
    assert made == 1
