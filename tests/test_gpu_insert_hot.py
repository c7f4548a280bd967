"""Inserts of more than 8,192 cells a table whose sets share a few buckets: the
batch goes to the full merge before anything of it is sorted, and a batch of the
same size without such buckets is merged slot by slot; both equal the oracle's."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2106_11565_gb300 import workloads as WL
from test_gpu_insert_delta import check, sets_slice

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_2106_11565_gb300 import _build, flinng
    _build.build()
    return flinng


@pytest.mark.parametrize("R,B,W,m", [(2, 300, 14, 4300), (4, 700, 15, 2100), (3, 200, 14, 4000)])
def test_hot_and_spread_batches(F, R, B, W, m):
    L, n0 = 6, 26_000
    n = n0 + 2 * m
    pts = WL.random_sets(81, n, 30_000, 3, 30)
    off, el = pts
    # the second batch: nine sets in ten are the same one
    lo = n0 + m
    rows = [np.array([4, 8, 15], np.uint32) if (i >= lo and i % 10) else el[off[i]:off[i + 1]] for i in range(n)]
    pts = WL.csr_from_rows(rows)
    q = WL.random_sets(82, 30, 30_000, 3, 30)
    dp = WL.doph_params(83, L, 1)
    ix = F.Index("jaccard", R, B, L, 1, capacity=n + m, params=dp, W=W)
    o = O.OracleIndex("jaccard", R, B, L, 1, W, doph=dp)
    launches = []
    for a, b in ((0, n0), (n0, lo), (lo, n)):
        part, perm = sets_slice(pts, a, b), WL.group_permutations(84 + a, R, b - a)
        c0 = F.kernel_launches()
        (ix.insert if a else ix.build)(part, perm)
        launches.append(F.kernel_launches() - c0)
        o.insert(part, perm)
    check(ix, o, q, o.hash(q))
    # a third of the index in one batch: the full merge, without a look at the partitions
    ix.close()
    full = F.Index("jaccard", R, B, L, 1, capacity=n0 + m, params=dp, W=W)
    full.build(sets_slice(pts, lo, lo + m), WL.group_permutations(90, R, m))
    c0 = F.kernel_launches()
    full.insert(sets_slice(pts, lo, n), WL.group_permutations(91, R, m))
    merge = F.kernel_launches() - c0
    full.close()
    assert launches[2] <= merge + 3, launches + [merge]
