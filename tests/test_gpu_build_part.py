"""The partitioned build from scratch at the sizes where its branches change,
against the oracle's reverse index: partitions of one bucket (W at or below the
coarse bits) and of the most buckets (W = coarse bits + 12), points around a
partition's and a CTA's capacity, lists sorted by a thread, a warp and a CTA,
buckets so full that their partition leaves shared memory (with lists above and
below the hot limit), every record width; R = 1 and W = 24 take the general
path."""
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


def draw_buckets(kind, rng, n, L, W):
    m = 1 << W
    if kind == "uniform":
        b = rng.integers(0, m, (n, L))
    elif kind == "clumped":                  # about 20 points a bucket
        b = rng.integers(0, m, (max(1, n // 20), L))[rng.integers(0, max(1, n // 20), n)]
    elif kind == "same":
        b = np.full((n, L), m - 1)
    else:                                    # hot: a third in one bucket, the rest Zipf-like
        b = np.minimum(m - 1, (m * rng.random((n, L)) ** 6).astype(np.int64))
        b[rng.random((n, L)) < 0.33] = m // 2
    return b.astype(np.uint32)


@pytest.mark.parametrize("kind", ["uniform", "clumped", "hot", "same"])
@pytest.mark.parametrize("n,L,W,R,B", [
    (1, 3, 5, 2, 7), (1024, 2, 13, 2, 300), (1537, 3, 9, 3, 40), (3073, 35, 1, 2, 33), (5000, 4, 17, 4, 1100),
    (9000, 5, 3, 8, 500), (20_000, 2, 20, 3, 4096), (40_000, 3, 6, 2, 9000), (700, 1, 24, 2, 50), (2500, 3, 10, 1, 90),
])
def test_csr_equals_oracle(F, n, L, W, R, B, kind):
    rng = np.random.default_rng([n, L, W])
    b = draw_buckets(kind, rng, n, L, W)
    perm = WL.group_permutations(3, R, n)
    ix = F.Index("jaccard", R, B, L, 1, capacity=n + 5, params=WL.doph_params(1, L, 1), W=W)
    ix.build_buckets(b[: (n + 1) // 2], WL.group_permutations(4, R, (n + 1) // 2))   # replaced below
    ix.build_buckets(b, perm)
    gid = np.zeros((n, R), np.uint16)
    O.groups(perm, B, 0, gid)
    off, cells = O.build_csr(b, gid, B, W)
    ex = ix.export()
    assert np.array_equal(ex["gid"], gid)
    assert np.array_equal(ex["off"], off) and np.array_equal(ex["cells"], cells)
    q = b[rng.integers(0, n, 12)]
    got = ix.counts(q)                       # heavy lists are read as bitmaps
    for i in range(12):
        assert np.array_equal(got[i], O.counts(off, cells, L, W, q[i], B * R))
    ix.close()


@pytest.mark.parametrize("universe,W,R,B", [(50_000, 14, 3, 300), (50_000, 20, 2, 5000), (400, 5, 4, 60), (3, 9, 3, 500),
                                            (9000, 9, 1, 200)])
def test_large_inserts_equal_oracle(F, universe, W, R, B):
    """Batches past the one-CTA-per-table limit: partitioned where their buckets
    spread, the full merge where many points share a bucket (a universe of three
    elements) or the batch outnumbers the index, R = 1 always."""
    L = 9
    sizes = [24_000, 5000, 9001, 30_000]
    N = sum(sizes)
    off, el = WL.random_sets(70 + W, N, universe, 1, min(universe, 40))
    dp = WL.doph_params(71, L, 1)
    ix = F.Index("jaccard", R, B, L, 1, capacity=N, params=dp, W=W)
    o = O.OracleIndex("jaccard", R, B, L, 1, W, doph=dp)
    lo = 0
    for step, n in enumerate(sizes):
        part = (off[lo:lo + n + 1] - off[lo]).astype(np.uint64), np.ascontiguousarray(el[off[lo]:off[lo + n]])
        perm = WL.group_permutations(72, R, n, batch=step)
        (ix.build if step == 0 else ix.insert)(part, perm)
        o.insert(part, perm)
        lo += n
        ex = ix.export()
        assert np.array_equal(ex["gid"], o.gid), step
        assert np.array_equal(ex["off"], o.off) and np.array_equal(ex["cells"], o.cells), step
        q = o.buckets[:: max(1, lo // 7)]
        got = ix.counts(q)
        for i in range(len(q)):
            assert np.array_equal(got[i], O.counts(o.off, o.cells, L, W, q[i], B * R)), step
    ix.close()
