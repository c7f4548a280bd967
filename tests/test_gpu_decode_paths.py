"""The decode's choices by size, against the oracle: few and many candidates at a
check (ranked directly up to 128, selected by digits above), floods of equal
scores that fill the candidate buffer, one and several records in flight (batches
resident at once, larger ones), cells of any size with and without the filter,
one repetition, and the gather's lists taken cell by cell."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2106_11565_gb300 import workloads as WL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_2106_11565_gb300 import _build, flinng
    _build.build()
    return flinng


@pytest.mark.parametrize("R,B,N,L", [(1, 60, 12_000, 40), (2, 300, 30_000, 8), (2, 500, 3000, 300), (3, 90, 9000, 20),
                                     (8, 200, 5000, 12)])
def test_floods(F, R, B, N, L):
    rng = np.random.default_rng([R, B, N])
    ix = F.Index("jaccard", R, B, 4, 1, capacity=N, params=WL.doph_params(1, 4, 1), W=6)
    ix.build(WL.random_sets(5, N, 500, 1, 4), WL.group_permutations(6, R, N))
    gid = ix.export()["gid"]
    moff, mem = O.members(gid, B)
    rows = [np.full(B * R, 1), rng.integers(0, 3, B * R), rng.integers(0, L + 1, B * R),
            np.where(rng.random(B * R) < 0.3, rng.integers(1, 4, B * R), 0),
            np.where(rng.random(B * R) < 0.05, L, 1)]
    rows = np.stack(rows).astype(np.uint16)
    for k in (1, 31, 32, 64, 127, 128, 129, 255, 256, 257, 513, 1024):
        want = [O.alg3(r, moff, mem, N, R, B, k, k_max=k) for r in rows]
        for nq in (5, 310, 1300):           # 512 threads, 256, 256 with 32 registers
            ids, sc = ix.query_counts(np.tile(rows, (nq // 5, 1)), k, L)
            for i in (0, 1, 2, 3, 4, nq - 5, nq - 3, nq - 1):
                assert np.array_equal(ids[i], want[i % 5][0]) and np.array_equal(sc[i], want[i % 5][1]), (k, nq, i)
    ix.close()


@pytest.mark.parametrize("R,B,N,L,W,size", [
    (2, 100, 3000, 16, 12, 90),      # a cell a list, a few hundred members a query
    (3, 40, 4000, 520, 12, 40),      # more tables than a round of any CTA
    (1, 150, 6000, 24, 5, 30),       # long lists, one repetition
    (2, 200, 9000, 9, 3, 8),         # nearly all members at the few scores there are
])
def test_batches(F, R, B, N, L, W, size):
    pts, q = WL.random_sets(71, N, 4000, 1, size), WL.random_sets(72, 1290, 4000, 0, size)
    dp = WL.doph_params(73, L, 1)
    perm = WL.group_permutations(74, R, N)
    ix = F.Index("jaccard", R, B, L, 1, capacity=N, params=dp, W=W)
    ix.build(pts, perm)
    o = O.OracleIndex("jaccard", R, B, L, 1, W, doph=dp)
    o.build(pts, perm)
    qb = o.hash(q)
    for k in (3, 100, 400):
        ids, sc = ix.query(q, k)             # 1,290 queries: 128 or 256 threads
        for m in (1290, 640, 320, 7):
            off = q[0][:m + 1]
            i2, s2 = ix.query((off, q[1][:int(off[-1])]), k)
            assert np.array_equal(i2, ids[:m]) and np.array_equal(s2, sc[:m]), (k, m)
            i2, s2 = ix.query_buckets(qb[:m], k)
            assert np.array_equal(i2, ids[:m]) and np.array_equal(s2, sc[:m]), (k, m)
        pick = np.r_[0:20, 600:620, 1270:1290]
        oid, osc = o.query_buckets(qb[pick], k)
        assert np.array_equal(ids[pick], oid) and np.array_equal(sc[pick], osc), k
    ix.close()
