"""MinHash values around the bin counts where the list of empty bins would cost
a resident CTA (and is left out), for sets shorter and longer than the bins, and
FP32 codes of short rows on both sides of the line between their kernels,
against the oracle."""
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


@pytest.mark.parametrize("L,K", [(33, 1), (455, 1), (1000, 1), (1365, 1), (1024, 2), (1025, 2), (1024, 4)])
def test_values(F, L, K):
    pts = WL.random_sets(91, 150, 60_000, 0, 900)
    dp = WL.doph_params(92, L, K)
    ix = F.Index("jaccard", 1, 1, L, K, capacity=1, params=dp, W=8)
    b, v, _ = ix.hash(pts, values=True)
    ref = O.doph(pts[0], pts[1], L * K, dp["doph_a"], dp["doph_b"], dp["doph_seed"])
    assert np.array_equal(v, ref)
    assert np.array_equal(b, O.minhash_buckets(ref, L, K, dp["bucket_a"], dp["bucket_c"], 8))
    ix.close()


@pytest.mark.parametrize("d,n", [(32, 1536), (32, 1537), (32, 3073), (127, 1537), (128, 3072), (128, 3073)])
def test_short_rows(F, d, n):
    L, K = 8, 8
    w = WL.srp_projections(93, L * K, d)
    x, _ = WL.gaussian_mixture(94, n, d, 9, 0.3)
    ix = F.Index("cosine", 1, 1, L, K, capacity=1, params=w, dim=d)
    assert np.array_equal(ix.hash(x)[0], O.srp_codes(x, w, L, K))
    ix.close()
