"""The SRP kernels at the sizes where their dispatch changes, against the
oracle's exact signs: small batches (a warp per projection) and larger ones (tiles
of 64 and of 128 rows), ragged rows, projections and dimensions, rows that 16-byte
loads cannot read, norms outside fp32's squared range, and the single-term
forms' dense second pass."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2106_11565_gb300 import workloads as WL
from test_gpu_tc_single import worst_case_error

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_2106_11565_gb300 import _build, flinng
    _build.build()
    return flinng


def rows(seed, n, d, w):
    x, _ = WL.gaussian_mixture(seed, n, d, 9, 0.3)
    for i in range(0, n, 6):                      # planted near-zero projections
        j = i % w.shape[0]
        if d > 1:
            x[i, -1] = np.float32(-float(np.dot(w[j, :-1].astype(np.float64), x[i, :-1])) / float(w[j, -1]))
    if n > 4:
        x[2] = 0.0
        x[3] *= np.float32(1e25)                  # squares overflow fp32
        x[4] *= np.float32(1e-28)                 # squares underflow
    return np.ascontiguousarray(x, np.float32)


@pytest.mark.parametrize("n", [1, 8, 9, 129, 192, 193, 1300])
@pytest.mark.parametrize("d,L,K,pad", [(1, 3, 7, 0), (33, 13, 5, 0), (100, 8, 8, 4), (100, 9, 7, 1), (516, 60, 17, 0), (36, 64, 16, 0)])
def test_fp32_codes(F, n, d, L, K, pad):
    import torch
    w = WL.srp_projections(400 + d, L * K, d)
    x = rows(500 + n, n, d, w)
    wide = torch.zeros((n, d + pad), dtype=torch.float32, device="cuda")
    wide[:, :d] = torch.from_numpy(x)
    ix = F.Index("cosine", 1, 1, L, K, capacity=1, params=w, dim=d)
    ocodes, oproj, _ = O.srp_codes(x, w, L, K, want_proj=True)
    codes, _, proj = ix.hash(wide, proj=True)
    assert np.array_equal(codes.cpu().numpy().view(np.uint32), ocodes)
    # n products in chains of any length: at most d roundings, 2 d u sum |w x|
    s = np.abs(x.astype(np.float64)) @ np.abs(w.astype(np.float64)).T
    assert np.all(np.abs(proj.cpu().numpy() - oproj) <= 2 * d * 2.0 ** -24 * s + d * 2.0 ** -146)
    ix.close()


@pytest.mark.parametrize("form", ["BF16X2", "BF16", "FP8"])
@pytest.mark.parametrize("n,d,L,K", [(5, 128, 16, 16), (96, 64, 64, 16), (97, 64, 5, 7), (1025, 256, 64, 16), (2100, 144, 33, 17)])
def test_tensor_core_codes(F, form, n, d, L, K):
    """n <= 96 without projections: the fp32 kernel; n * L * K >= 2^20: the
    dense second pass."""
    w = WL.srp_projections(600 + d, L * K, d)
    x = rows(700 + n, n, d, w)
    ix = F.Index("cosine", 1, 1, L, K, capacity=1, params=w, dim=d, precision=getattr(F, "PREC_" + form))
    codes, _, _ = ix.hash(x)
    assert np.array_equal(codes, O.srp_codes(x, w, L, K))
    cnt = ix.hash_counters()
    assert cnt["undecided"] >= 1 and cnt["flips"] <= cnt["undecided"]
    if n > 96:
        assert cnt["compensated"] == cnt["undecided"]
    # projections, from the dense pass's kernel too: within the formats' worst case
    codes, _, proj = ix.hash(x, proj=True)
    ocodes, oproj, _ = O.srp_codes(x, w, L, K, want_proj=True)
    assert np.array_equal(codes, ocodes)
    if form != "BF16X2":
        assert np.all(np.abs(proj - oproj) <= worst_case_error(x, w, form.lower()) * 1.01)
    ix.close()
