"""Per-cell counts written and read eight at a time, against the oracle: cell
totals that are and are not multiples of eight, output and input rows off a
16-byte boundary, 8- and 16-bit counters, counts above the largest allowed one
(clamped)."""
import ctypes as C

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


@pytest.mark.parametrize("L", [7, 255, 256])
@pytest.mark.parametrize("R,B", [(1, 8), (1, 3), (2, 4), (3, 100), (2, 1024), (3, 4097)])
@pytest.mark.parametrize("shift", [0, 1, 4])
def test_counts_out_and_in(F, L, R, B, shift):
    import torch
    n = 2 * B + 5
    pts = WL.random_sets(70 + L + B, n, 300, 5, 20)
    q = WL.random_sets(71 + L + B, 9, 300, 5, 20)
    dp = WL.doph_params(72 + L, L, 1)
    ix = F.Index("jaccard", R, B, L, 1, capacity=n, params=dp, W=6)
    perm = WL.group_permutations(73 + L, R, n)
    ix.build(pts, perm)
    o = O.OracleIndex("jaccard", R, B, L, 1, 6, doph=dp)
    o.build(pts, perm)
    qv = O.doph(q[0], q[1], L, dp["doph_a"], dp["doph_b"], dp["doph_seed"])
    qb = O.minhash_buckets(qv, L, 1, dp["bucket_a"], dp["bucket_c"], 6)
    ref = np.stack([O.counts_direct(o.buckets, o.gid, B, row) for row in qb])
    buf = torch.full((9 * B * R + 16,), 0x5A5A, dtype=torch.int16, device="cuda")
    out = buf[shift:shift + 9 * B * R]
    qd = torch.from_numpy(qb.view(np.int32)).cuda()
    F._check(ix.lib.flinng_counts(ix.h, C.c_void_p(qd.data_ptr()), 9, C.c_void_p(out.data_ptr()), 1))
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy().view(np.uint16).reshape(9, -1), ref)
    assert torch.all(buf[:shift] == 0x5A5A) and torch.all(buf[shift + 9 * B * R:] == 0x5A5A)
    # read back from the same place; counts over L count as L
    big = ref.astype(np.int64) + np.where(np.arange(B * R) % 5 == 0, 40000, 0)
    out.copy_(torch.from_numpy(big.astype(np.uint16).view(np.int16).ravel()).cuda())
    ids, sc = ix.query_counts(out.view(9, B * R), 5, L)
    want = np.minimum(big, L).astype(np.uint16)
    moff, mem = O.members(o.gid, B)
    for i in range(9):
        oids, osc, _ = O.alg3(want[i], moff, mem, n, R, B, 5, k_max=5)
        assert np.array_equal(ids[i].cpu().numpy().view(np.uint32), oids)
        assert np.array_equal(sc[i].cpu().numpy().view(np.uint16), osc)
    ix.close()
