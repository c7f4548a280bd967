"""Query shapes near the limit of a CTA's shared memory: where 512 threads (the
usual choice) do not fit, 256 or 128 do, and where no fused shape does, the
batch is hashed first. Every form of the call takes them, with the answers of
the bucket call, which hashes nothing."""
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


def check(F, ix, q, dq, k):
    import torch
    buckets = ix.hash(q)[0]
    want, wsc = ix.query_buckets(buckets, k)
    nq = want.shape[0]

    def same(ids, sc):
        torch.cuda.synchronize()
        sc = sc.cpu().numpy() if hasattr(sc, "is_cuda") else sc
        assert np.array_equal(u32(ids), want) and np.array_equal(sc.view(np.uint16), wsc)

    for mode in (F.QUERY_PLAIN, F.QUERY_FUSED, F.QUERY_GRAPH):
        ix.set_query_mode(mode)
        same(*ix.query(q, k))
        same(*ix.query(dq, k))
    ix.set_query_mode(F.QUERY_FUSED)
    for threads in (128, 256, 512):
        ix.set_tuning(nq, threads)
        same(*ix.query(dq, k))
    ix.tune(dq, k)
    same(*ix.query(dq, k))
    srv = F.Server(hbm_budget=8 << 30, n_slots=2, max_batch=4, k_max=k)
    which = srv.add_index(ix)
    reqs = np.zeros(nq, F.REQ_DTYPE)
    reqs["kind"], reqs["index"], reqs["k"] = F.REQ_QUERY, which, k
    if ix.metric == "cosine":
        reqs["n"] = q.shape[1]
        reqs["data"] = q.ctypes.data + np.arange(nq, dtype=np.uint64) * np.uint64(4 * q.shape[1])
    else:
        reqs["n"] = np.diff(q[0])
        reqs["data"] = q[1].ctypes.data + q[0][:-1] * np.uint64(4)
    ids, sc, _ = srv.replay(reqs)
    same(ids, sc)
    srv.close()


# 512 threads alone too large; 256 too; only the form that hashes first
@pytest.mark.parametrize("R,B,L,k", [(8, 8192, 4095, 10), (8, 8191, 3900, 512), (8, 8192, 4095, 512)])
def test_sets(F, R, B, L, k):
    import torch
    N, nq = 9000, 7
    pts, q = WL.random_sets(41, N, 3000, 2, 20), WL.random_sets(42, nq, 3000, 2, 20)
    ix = F.Index("jaccard", R, B, L, 1, capacity=N, params=WL.doph_params(43, L, 1), W=3)
    ix.build(pts, WL.group_permutations(44, R, N))
    dq = (torch.from_numpy(q[0].view(np.int64)).cuda(), torch.from_numpy(q[1].view(np.int32)).cuda())
    check(F, ix, q, dq, k)
    ix.close()


@pytest.mark.parametrize("R,B,L,d,k", [(3, 2000, 5, 50_000, 10), (8, 2273, 2, 50_088, 100), (4, 956, 5, 52_428, 512)])
def test_vectors(F, R, B, L, d, k):
    import torch
    N, nq = 6000, 5
    rng = np.random.default_rng([R, B])
    pts = rng.standard_normal((N, d), dtype=np.float32)
    q = np.ascontiguousarray(pts[rng.integers(0, N, nq)] + np.float32(0.3) * rng.standard_normal((nq, d), dtype=np.float32))
    ix = F.Index("cosine", R, B, L, 1, capacity=N, params=WL.srp_projections(45, L, d), dim=d)
    ix.build(torch.from_numpy(pts).cuda(), torch.from_numpy(WL.group_permutations(46, R, N).view(np.int32)).cuda())
    check(F, ix, q, torch.from_numpy(q).cuda(), k)
    ix.close()
