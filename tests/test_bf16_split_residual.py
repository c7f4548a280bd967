"""The two-term BF16 split's margin from measured residual norms, against fp64
(no GPU): for rows x = x1 + r_x and w = w1 + r_w with x1 = bf16(x), x2 =
bf16(r_x), the terms x1.w1 + x1.w2 + x2.w1 miss x.w by at most
2^-8 (|x| |r_w| + |r_x| |w|) + (1 + 2^-6) |r_x| |r_w| (norms), whatever the
rows: random ones, ones one unit beside bf16 ties (the largest residuals),
exact bf16 values (none), one large entry among small ones, aligned residuals
of one sign."""
import numpy as np
import pytest

from test_bf16_split_bound import split


def rows(kind, rng, d):
    if kind == "ties":
        u = (rng.integers(0x3F000000, 0x41000000, d, dtype=np.uint64) & 0xFFFF0000) | 0x7FFF
        return u.astype(np.uint32).view(np.float32)
    if kind == "exact":
        return split(rng.standard_normal(d))[0]
    x = rng.standard_normal(d).astype(np.float32)
    if kind == "spike":
        x *= np.float32(1e-3)
        x[0] = np.float32(1000.3)
    return x


@pytest.mark.parametrize("kx", ["normal", "ties", "exact", "spike"])
@pytest.mark.parametrize("kw", ["normal", "ties", "exact", "spike"])
@pytest.mark.parametrize("d", [8, 128, 4096])
def test_dropped_sum_within_residual_norms(kx, kw, d):
    rng = np.random.default_rng(d + len(kx) * 7 + len(kw))
    for _ in range(20):
        x, w = rows(kx, rng, d), rows(kw, rng, d)
        if d == 8:
            w = np.copysign(w, x).astype(np.float32)      # nothing cancels
        x1, x2, _ = (np.asarray(v, np.float64) for v in split(x))
        w1, w2, _ = (np.asarray(v, np.float64) for v in split(w))
        x, w = x.astype(np.float64), w.astype(np.float64)
        # term by term: the products are exact in fp64 and the large parts cancel
        miss = abs(np.sum(x * w - (x1 * w1 + x1 * w2 + x2 * w1)))
        nx, nw, rx, rw = (np.linalg.norm(v) for v in (x, w, x - x1, w - w1))
        bound = 2.0 ** -8 * (nx * rw + rx * nw) + (1 + 2.0 ** -6) * rx * rw
        assert miss <= bound + d * 2.0 ** -52 * nx * nw
        if kx == kw == "exact":
            assert bound == 0.0
