"""Index construction on a device with little room left: the tensor-core
assignment's operands (as large as the rows) are done without, down to what the
FP32 kernel needs, and the lists are the same."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.mark.parametrize("spare", [120, 280])  # MB beside the index's rows: below the operands', below theirs and the k-means' rows
def test_build_without_room_for_the_operands(spare):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    rt = C.CDLL("libcudart.so.13")
    rt.cudaMalloc.argtypes, rt.cudaFree.argtypes = [C.POINTER(C.c_void_p), C.c_size_t], [C.c_void_p]
    g = torch.Generator(device="cuda").manual_seed(2)
    X = (8 * torch.rand((400_000, 128), generator=g, device="cuda")).round()  # 205 MB; operands 234 MB, k-means rows 67 MB

    def build():
        ix = ksc.build_index(X, 512, 64, iters=2, seed=3)
        e = ix.export(fields=("assign", "codes"))
        ix.free()
        return e["assign"], e["codes"]

    want = build()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held, left = [], 205 * MB + spare * MB
    try:
        for size in (8 << 30, 512 * MB, 16 * MB, 2 * MB):
            while torch.cuda.mem_get_info()[0] >= left + size:
                p = C.c_void_p()
                if rt.cudaMalloc(C.byref(p), size):
                    break
                held.append(p)
        assert left <= torch.cuda.mem_get_info()[0] < left + 8 * MB
        got = build()
    finally:
        for p in held:
            assert rt.cudaFree(p) == 0
    for a, b in zip(want, got):
        np.testing.assert_array_equal(a, b)
