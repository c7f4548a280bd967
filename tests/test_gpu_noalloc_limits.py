"""Batches that flinng_query_noalloc takes in the single-term tensor-core
precisions: one byte (FP8) or two (BF16) of scratch per coordinate and 16 per
projection, whatever the hash does inside; the answers are flinng_query's."""
import ctypes as C

import numpy as np
import pytest

from paper_2106_11565_gb300 import workloads as WL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_2106_11565_gb300 import _build, flinng
    _build.build()
    return flinng


@pytest.mark.parametrize("form,d,L,K,most", [
    ("FP8", 4096, 8, 8, 1017), ("FP8", 4096, 64, 16, 255), ("FP8", 64, 8, 8, 4707), ("BF16", 4096, 8, 8, 566),
    ("BF16", 256, 16, 16, 1130), ("BF16", 64, 8, 8, 4450), ("BF16X2", 4096, 8, 8, 300),
])
def test_limits(F, form, d, L, K, most):
    import torch
    N, R, k = 2000, 2, 10
    pts, _ = WL.gaussian_mixture(51, N, d, 30, 0.2)
    ix = F.Index("cosine", R, 50, L, K, capacity=N, params=WL.srp_projections(52, L * K, d), dim=d,
                 precision=getattr(F, "PREC_" + form))
    ix.build(pts, WL.group_permutations(53, R, N))

    def call(nq):
        q = torch.from_numpy(WL.noisy_queries(54, pts, nq, 0.1)[0]).cuda()
        fp, n, dev, keep = ix._points(q)
        ids = torch.full((nq, k), 7, dtype=torch.int32, device="cuda")
        sc = torch.full((nq, k), 7, dtype=torch.int16, device="cuda")
        rc = F.load().flinng_query_noalloc(ix.h, C.byref(fp), nq, None, k, ids.data_ptr(), sc.data_ptr())
        torch.cuda.synchronize()
        return rc, q, ids, sc

    for nq in (most, most // 3, 1):
        rc, q, ids, sc = call(nq)
        assert rc == F.OK, F.load().flinng_last_error()
        want, wsc = ix.query(q, k)
        torch.cuda.synchronize()
        assert torch.equal(ids, want) and torch.equal(sc, wsc)
    # one more is refused
    assert call(most + 1)[0] == F.ERR_INVALID_ARG
    ix.close()
