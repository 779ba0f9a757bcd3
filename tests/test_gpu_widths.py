"""Kernels chosen by width against the oracle, bit for bit (arXiv 2608.07152
Sec. 2.1, 2.3.1): the interval pass at every multiple of 64 bytes it holds the
query for in registers and past it, and the allocation-free ranking at the
edges of its loads (16-byte or scalar) and of its blocks' keys."""
import numpy as np
import pytest
import torch

import paper_2608_07152_gb300 as pvs
from oracle import pvs_oracle as po

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", range(1, 19))
def test_bounds_at_every_width(k):
    m, n = 64 * k - (k % 3) * 21, 333       # 64 k bytes a row: whole and ragged
    rng = np.random.default_rng(k)
    V = rng.standard_normal((n, m)).astype(np.float32)
    q = rng.standard_normal(m).astype(np.float32)
    index = pvs.pvs_build(V)
    try:
        cur = pvs.pvs_cursor_open(index, q)
        try:
            lo, hi = pvs.pvs_cursor_bounds(cur, 0, n)
        finally:
            pvs.pvs_cursor_close(cur)
    finally:
        pvs.pvs_index_free(index)
    ref_lo, ref_hi = po.intervals(po.encode_query(q), po.quantize(V), m)
    assert np.array_equal(lo.view(np.uint32), ref_lo.view(np.uint32))
    assert np.array_equal(hi.view(np.uint32), ref_hi.view(np.uint32))


@pytest.mark.parametrize("n", [1, 31, 33, 1_000, 2_048, 2_049, 8_192])
@pytest.mark.parametrize("dim,offset", [(1, 0), (3, 0), (4, 0), (4, 1), (255, 0), (256, 0),
                                        (257, 0), (768, 0), (768, 1), (772, 0), (1_541, 0)])
def test_noalloc_ranking_at_its_edges(n, dim, offset):
    rng = np.random.default_rng(n + dim)
    V = rng.standard_normal((n, dim)).astype(np.float32)
    q = rng.standard_normal(dim).astype(np.float32)
    V[: n // 4] = V[n // 4: 2 * (n // 4)]                     # ties by id
    V[n // 2: n // 2 + n // 8, : dim // 2] *= np.float32(2.0 ** 40)
    V[n - n // 8:] = 0
    if dim > 1:                                               # exact cancellation
        q[1] = q[0]
        V[n // 3, :2] = (3e10, -3e10)
    flat = torch.zeros(n * dim + 4, device="cuda")
    Vd = flat[offset:offset + n * dim].view(n, dim)           # 4 bytes off the boundary
    Vd.copy_(torch.from_numpy(V))
    top = max(1, n - n // 3)
    ids = torch.empty(top, dtype=torch.int64, device="cuda")
    sc = torch.empty(top, dtype=torch.float32, device="cuda")
    pvs.pvs_rank_exact_noalloc(torch.from_numpy(q).cuda(), Vd, top, ids, sc)
    ref_ids, ref_sc = po.dense_ranking(q, V)
    assert np.array_equal(ids.cpu().numpy(), ref_ids[:top])
    assert np.array_equal(sc.cpu().numpy().view(np.uint32), ref_sc[:top].view(np.uint32))
