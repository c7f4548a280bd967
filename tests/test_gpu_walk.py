"""The decode's walk at the sizes where its branches change, against the
oracle's Alg. 3 on the same per-cell counts: cells of fewer than eight members
(one member per lane), eight and more (units of eight with ragged ends), one
cell of all points, empty cells; levels larger than the level list (2,048
cells), whole-range levels, a filter that passes few or most members, floods of
equal scores (buffer compaction), 8- and 16-bit counts, every record width."""
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


def counts_of(kind, rng, BR, L):
    if kind == "flat":                       # one level holds every cell
        return np.full(BR, max(1, L // 2))
    if kind == "two":                        # two levels of about half the cells each
        return rng.integers(1, 3, BR)
    if kind == "sparse":                     # almost all below t_min
        c = np.zeros(BR, np.int64)
        hit = rng.choice(BR, max(1, BR // 50), replace=False)
        c[hit] = rng.integers(1, L + 1, hit.size)
        return c
    if kind == "noise":                      # few high cells over a floor of ties
        return np.minimum(L, rng.geometric(0.5, BR) - 1 + L // 2 * (rng.random(BR) < 0.01))
    return rng.integers(0, L + 1, BR)        # uniform over the levels


@pytest.mark.parametrize("R,B,N,L,design", [
    (1, 3000, 20_000, 16, "even"), (2, 40, 1500, 255, "even"), (2, 5000, 45_000, 12, "even"),
    (3, 2049, 16_500, 256, "even"), (3, 2048, 2000, 30, "even"), (4, 700, 6000, 64, "uneven"),
    (4, 300, 9000, 20, "one"), (8, 900, 8100, 600, "uneven"),
])
def test_walk_equals_alg3(F, R, B, N, L, design):
    rng = np.random.default_rng([R, B, N])
    if design == "even":
        g = np.stack([(np.argsort(rng.permutation(N)) % B) for _ in range(R)])
    elif design == "uneven":                 # groups of very different sizes, some empty
        g = np.minimum(B - 1, (B * rng.random((R, N)) ** 3).astype(np.int64))
    else:                                    # every point in one group of repetition 0
        g = rng.integers(0, B, (R, N))
        g[0] = 7
    g = g.astype(np.uint16)
    pts = WL.random_sets(5, N, 500, 1, 4)
    ix = F.Index("jaccard", R, B, 4, 1, capacity=N, params=WL.doph_params(1, 4, 1), W=6)
    ix.build_groups(pts, g)
    gid = O.design_groups(g, B)
    moff, mem = O.members(gid, B)
    kinds = ["flat", "two", "sparse", "noise", "uniform"]
    cnt = np.stack([counts_of(k, rng, B * R, L) for k in kinds]).astype(np.uint16)
    for k_max in (1, 10, 129, 1024):
        k = np.array([k_max, max(1, k_max // 2), k_max, k_max, min(3, k_max)], np.uint32)
        ids, sc = ix.query_counts(cnt, k_max, L, k=k)
        for i, kind in enumerate(kinds):
            oid, osc, _ = O.alg3(cnt[i], moff, mem, N, R, B, int(k[i]), k_max=k_max)
            assert np.array_equal(ids[i], oid) and np.array_equal(sc[i], osc), (kind, k_max)
    ix.close()


@pytest.mark.parametrize("L,K,W,B", [(5, 1, 9, 33), (300, 1, 8, 2500), (16, 2, 4, 64)])
@pytest.mark.parametrize("threads,cap", [(128, 0), (256, 512), (512, 0)])
def test_gather_and_fused_shapes(F, L, K, W, B, threads, cap):
    """Lists that start and end anywhere in their 16-byte units, heavy and
    light, counted and decoded in the fused kernel at every CTA size."""
    R, N = 3, 4000
    pts = WL.random_sets(21 + L, N, 3000, 5, 90)
    q = WL.random_sets(22 + L, 70, 3000, 5, 90)
    dp = WL.doph_params(23, L, K)
    perm = WL.group_permutations(24, R, N)
    ix = F.Index("jaccard", R, B, L, K, capacity=N, params=dp, W=W)
    ix.build(pts, perm)
    o = O.OracleIndex("jaccard", R, B, L, K, W, doph=dp)
    o.build(pts, perm)
    ix.set_tuning(70, threads, 0, cap)
    for k in (1, 37, 300):
        ids, sc = ix.query(q, k)
        oid, osc = o.query(q, k)
        assert np.array_equal(ids, oid) and np.array_equal(sc, osc), k
    qb = o.hash(q)
    cnt = ix.counts(qb)
    for i in range(0, 70, 9):
        assert np.array_equal(cnt[i], O.counts(o.off, o.cells, L, W, qb[i], B * R))
    ix.close()
