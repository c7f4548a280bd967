"""FP32 signs where the sums leave the normal range: rows so small that a
factor of the margin would underflow, and sums that overflow on the way although
the row's norm does not, against the oracle's exact signs."""
import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_2106_11565_gb300 import _build, flinng
    _build.build()
    return flinng


def same_codes(F, x, w, L, K):
    ix = F.Index("cosine", 1, 1, L, K, capacity=1, params=w, dim=x.shape[1])
    ref = O.srp_codes(x, w, L, K)
    for n in (x.shape[0], 300, 20):                 # tiles of 128 and of 64 rows, a warp per projection
        codes = ix.hash(x[:n])[0]
        bad = np.argwhere(codes != ref[:n])
        assert bad.size == 0, (n, len(bad), bad[:4])
    ix.close()


@pytest.mark.parametrize("d", [24, 100])
def test_tiny_rows_and_large_projections(F, d):
    rng = np.random.default_rng(d)
    L, K, n = 64, 16, 1300
    w = (rng.standard_normal((L * K, d)) * 1e12).astype(np.float32)
    x = (rng.standard_normal((n, d)) * 3e-41).astype(np.float32)
    for j in range(L * K):                          # w_j . x_j nearly cancels
        i = j % n
        rest = float(np.dot(w[j, :-1].astype(np.float64), x[i, :-1].astype(np.float64)))
        w[j, -1] = np.float32(-rest / float(x[i, -1]))
    same_codes(F, x, w, L, K)


@pytest.mark.parametrize("d", [8, 36])
def test_sums_that_overflow(F, d):
    rng = np.random.default_rng(100 + d)
    L, K, n = 64, 16, 1300
    x = np.zeros((n, d), np.float32)
    x[:, :8] = 1e38 * rng.uniform(0.9, 1.1, (n, 8))
    x[:, 8:] = 1e36 * rng.standard_normal((n, d - 8))
    w = rng.standard_normal((L * K, d)).astype(np.float32)
    w[:, :4] = 4.0                                  # four products past the largest float,
    w[:, 4:8] = -4.0                                # then four of the other sign
    w[:, :8] *= np.float32(1) + np.float32(0.05) * rng.standard_normal((L * K, 1)).astype(np.float32)
    same_codes(F, x, w, L, K)
