"""Ranking of rows wider than 256: the 16-bit tensor-core scores only preselect
lists for the exact FP32 ranking, so the ranked lists are those of the exact
distances also where the scores say nothing (centroids far from the origin and
close together) and where more lists are left than the re-score buffer holds.
Coordinates lie on a grid of 1/16, so FP32 distances are exact and the order
(ties to the lower list) is known."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,L", [(512, 40), (512, 1024), (512, 1025), (320, 2048), (258, 1500)])
@pytest.mark.parametrize("offset", [0, 20, 400])
def test_wide_rows_ranked_exactly(d, L, offset):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    rng = np.random.default_rng(d + L + offset)
    C = (offset + rng.integers(-64, 65, size=(L, d)) / 16.0).astype(np.float32)
    Q = (offset + rng.integers(-64, 65, size=(400, d)) / 16.0).astype(np.float32)
    M = d // 2 if d < 512 else d // 4
    ix = ksc.index_import(dict(X=C, c_rank=C, c_mean=C, codebook=np.zeros((M, 16, d // M), np.float32),
                               codes=np.zeros((L, M), np.uint8), assign=np.arange(L, dtype=np.int32)))
    # whole numbers of 1/256 below 2^24 (in FP32) and 2^53 (here)
    q, c = np.rint(16 * Q.astype(np.float64)), np.rint(16 * C.astype(np.float64))
    D = (q * q).sum(1)[:, None] + (c * c).sum(1)[None] - 2 * q @ c.T
    P = 20
    want = np.argsort(D, axis=1, kind="stable")[:, :P]
    probes, scores = ix.rank_lists(torch.from_numpy(Q).cuda(), P)
    np.testing.assert_array_equal(probes.cpu().numpy(), want)
    np.testing.assert_array_equal(scores.cpu().numpy(), (np.take_along_axis(D, want, 1) / 256).astype(np.float32))


@pytest.mark.parametrize("scale", [1, 1000, 4000, 8000])
def test_operand_types(scale):
    """Centroids whose norms, or coordinates, pass what the FP16 operands take."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_03298_gb300 import ksc
    rng = np.random.default_rng(scale)
    C = (scale * rng.integers(-3, 4, size=(300, 64))).astype(np.float32)
    Q = (scale * rng.integers(-3, 4, size=(400, 64))).astype(np.float32)
    ix = ksc.index_import(dict(X=C, c_rank=C, c_mean=C, codebook=np.zeros((16, 16, 4), np.float32),
                               codes=np.zeros((300, 16), np.uint8), assign=np.arange(300, dtype=np.int32)))
    q, c = Q.astype(np.float64) / scale, C.astype(np.float64) / scale
    D = (q * q).sum(1)[:, None] + (c * c).sum(1)[None] - 2 * q @ c.T
    probes, _ = ix.rank_lists(torch.from_numpy(Q).cuda(), 10)
    np.testing.assert_array_equal(probes.cpu().numpy(), np.argsort(D, axis=1, kind="stable")[:, :10])
