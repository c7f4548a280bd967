"""Levels of more cells than the level list holds (2,048), at the counts whose
level cursors lie where the decode's chunk scratch ends (twice the CTA's
threads: 256, 512, 1,024, 2,048) and next to them, against the oracle."""
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


@pytest.mark.parametrize("R,B,N", [(2, 2500, 9000), (3, 6000, 14_000), (1, 4500, 4500)])
def test_given_counts(F, R, B, N):
    rng = np.random.default_rng([R, B])
    perm = WL.group_permutations(3, R, N)
    ix = F.Index("jaccard", R, B, 4, 1, capacity=N, params=WL.doph_params(1, 4, 1), W=6)
    ix.build(WL.random_sets(5, N, 500, 1, 4), perm)
    gid = ix.export()["gid"]
    moff, mem = O.members(gid, B)
    for L in (512, 1024, 2048, 4095):
        cnt = []
        for t in (256, 511, 512, 1024, 2047, 2048):
            if t > L:
                continue
            cnt.append(np.full(B * R, t))
            c = np.full(B * R, t)                     # one cell in ten elsewhere
            hit = rng.random(B * R) < 0.1
            c[hit] = rng.integers(0, L + 1, hit.sum())
            cnt.append(c)
        cnt = np.stack(cnt).astype(np.uint16)
        for k in (1, 100, 700):
            ids, sc = ix.query_counts(cnt, k, L)
            for i in range(len(cnt)):
                oid, osc, _ = O.alg3(cnt[i], moff, mem, N, R, B, k, k_max=k)
                assert np.array_equal(ids[i], oid) and np.array_equal(sc[i], osc), (L, k, i)
    ix.close()


@pytest.mark.parametrize("threads", [0, 128, 256, 512])
@pytest.mark.parametrize("L", [256, 512, 1024])
def test_equal_sets(F, L, threads):
    """Every stored set the same: a query of it meets all cells at count L."""
    R, B, N, W = 2, 2500, 3000, 6
    off = (np.arange(N + 1) * 3).astype(np.uint64)
    el = np.tile(np.array([5, 77, 901], np.uint32), N)
    dp = WL.doph_params(9, L, 1)
    perm = WL.group_permutations(4, R, N)
    ix = F.Index("jaccard", R, B, L, 1, capacity=N, params=dp, W=W)
    ix.build((off, el), perm)
    o = O.OracleIndex("jaccard", R, B, L, 1, W, doph=dp)
    o.build((off, el), perm)
    q = (off[:41], el[:120])
    if threads:
        ix.set_tuning(40, threads)
    for k in (1, 100):
        ids, sc = ix.query(q, k)
        oid, osc = o.query((off[:2], el[:3]), k)
        assert np.array_equal(ids, np.repeat(oid, 40, 0)) and np.array_equal(sc, np.repeat(osc, 40, 0))
        ids, sc = ix.query_buckets(o.hash(q), k)
        assert np.array_equal(ids[17], oid[0]) and np.array_equal(sc[17], osc[0])
    ix.close()
