"""Host query vectors in page-locked memory that a copy queued on the index's
stream has yet to fill: the query reads them in stream order."""
import numpy as np
import pytest

from paper_2106_11565_gb300 import workloads as WL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_2106_11565_gb300 import _build, flinng
    _build.build()
    return flinng


@pytest.mark.parametrize("nq,d", [(1, 64), (30, 40), (400, 64)])
@pytest.mark.parametrize("mode", [1, 2])
def test_vectors_filled_by_a_queued_copy(F, nq, d, mode):
    import torch
    N, L, K, R = 1000, 8, 6, 2
    pts, _ = WL.gaussian_mixture(61, N, d, 20, 0.2)
    q, _ = WL.noisy_queries(62, pts, nq, 0.1)
    ix = F.Index("cosine", R, 30, L, K, capacity=N, params=WL.srp_projections(63, L * K, d), dim=d)
    ix.build(pts, WL.group_permutations(64, R, N))
    ix.set_query_mode(mode)
    want, wsc = ix.query(q, 20)
    dev = torch.from_numpy(q).cuda()
    host = torch.zeros((nq, d), dtype=torch.float32).pin_memory()
    view = host.numpy()
    ix.query(view, 20)                              # shapes and graphs laid out
    host.zero_()
    torch.cuda._sleep(20_000_000)                   # about 10 ms of work before the copy
    host.copy_(dev, non_blocking=True)
    ids, sc = ix.query(view, 20)
    assert np.array_equal(ids, want) and np.array_equal(sc, wsc)
    ix.close()
