"""Host queries around the size of the index's pinned staging (64 KB of inputs
and outputs): below it the kernel works in the staging, above it the buffers
are copied; both equal the device-buffer call, in every query mode, with ragged
k, padded rows and without elements."""
import numpy as np
import pytest

from paper_2106_11565_gb300 import workloads as WL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_2106_11565_gb300 import _build, flinng
    _build.build()
    return flinng


def u32(a):
    return (a.cpu().numpy() if hasattr(a, "is_cuda") else np.asarray(a)).view(np.uint32)


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("nq,k", [(1, 1), (1, 1024), (13, 100), (40, 200), (60, 200), (700, 3)])
def test_sets(F, mode, nq, k):
    import torch
    N, L, R = 1500, 24, 3
    pts, q = WL.random_sets(31, N, 2000, 5, 80), WL.random_sets(32, nq, 2000, 0, 80)
    ix = F.Index("jaccard", R, 50, L, 1, capacity=N, params=WL.doph_params(33, L, 1), W=10)
    ix.build(pts, WL.group_permutations(34, R, N))
    ix.set_query_mode(mode)
    kk = ((np.arange(nq) * 37) % (k + 1)).astype(np.uint32)
    el = q[1] if len(q[1]) else np.zeros(1, np.uint32)
    dq = (torch.from_numpy(q[0].view(np.int64)).cuda(), torch.from_numpy(el.view(np.int32)).cuda())
    for kq in (None, kk):
        ids, sc = ix.query(q, k, k=kq)
        dids, dsc = ix.query(dq, k, k=None if kq is None else torch.from_numpy(kq.view(np.int32)).cuda())
        torch.cuda.synchronize()
        assert np.array_equal(u32(ids), u32(dids)) and np.array_equal(sc, dsc.cpu().numpy())
    ix.close()


@pytest.mark.parametrize("nq,d,pad", [(1, 40, 0), (30, 40, 3), (400, 40, 0), (409, 40, 0), (9, 1000, 24)])
def test_vectors(F, nq, d, pad):
    import torch
    N, L, K, R = 1000, 8, 6, 2
    pts, _ = WL.gaussian_mixture(35, N, d, 20, 0.2)
    q, _ = WL.noisy_queries(36, pts, nq, 0.1)
    wide = np.full((nq, d + pad), 7.0, np.float32)
    wide[:, :d] = q
    ix = F.Index("cosine", R, 30, L, K, capacity=N, params=WL.srp_projections(37, L * K, d), dim=d)
    ix.build(pts, WL.group_permutations(38, R, N))
    ids, sc = ix.query(wide, 20)
    dids, dsc = ix.query(torch.from_numpy(q).cuda(), 20)
    torch.cuda.synchronize()
    assert np.array_equal(u32(ids), u32(dids)) and np.array_equal(sc, dsc.cpu().numpy())
    ix.close()
