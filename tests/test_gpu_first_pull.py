"""The first pull of a lone cursor (the first working set scored and sorted
whole; arXiv 2608.07152 Sec. 2.1, 2.3.1) against the oracle: at the edges of
its sizes, and where its set is too large and the incremental pulls take over."""
import numpy as np
import pytest

import paper_2608_07152_gb300 as pvs
from oracle import pvs_oracle as po

pytestmark = pytest.mark.gpu


def _corpus(kind, n, m, rng):
    V = rng.standard_normal((n, m)).astype(np.float32)
    if kind == "clusters":      # about 500 near neighbours of the query
        V[: n // 8] = V[0] + 0.3 * V[: n // 8]
    elif kind == "alike":       # every interval holds every threshold
        V = (V[0] + 1e-3 * V).astype(np.float32)
    elif kind == "tied":        # exact ties across the whole set
        V = V[rng.integers(0, 7, n)]
    elif kind == "outlier":     # one score far above the rest
        V[n // 2] *= 1000.0
    return np.ascontiguousarray(V)


# visible counts around the horizon (2,048), sets around a sort's sizes (1,024,
# 4,096 rows; ties that no threshold splits) and the largest one scored whole
# (16,384), row counts around the values one CTA stages (51,200)
# and the per-slot bounds (from 48,640 rows on)
@pytest.mark.parametrize("kind,n,m", [
    ("iid", 1, 16), ("iid", 1_023, 64), ("iid", 2_048, 64), ("iid", 2_049, 33),
    ("iid", 4_097, 128), ("iid", 20_000, 32), ("clusters", 40_001, 96), ("iid", 51_201, 64),
    ("clusters", 60_003, 128), ("alike", 4_096, 64), ("alike", 4_097, 64), ("alike", 16_384, 64), ("alike", 16_385, 64),
    ("alike", 60_003, 64), ("tied", 9_001, 48),
    ("tied", 30_001, 48), ("outlier", 30_001, 48)])
@pytest.mark.parametrize("deleted", [0.0, 0.3, 0.7])
def test_pages_equal_the_oracle(kind, n, m, deleted):
    rng = np.random.default_rng(n + m)
    V = _corpus(kind, n, m, rng)
    q = (V[0] + 0.5 * rng.standard_normal(m)).astype(np.float32)
    vis = None
    index = pvs.pvs_build(V)
    try:
        if deleted:
            dead = np.flatnonzero(rng.random(n) < deleted)
            vis = np.ones(n, bool)
            vis[dead] = False
            pvs.pvs_tombstone(index, dead)
        ref_ids, ref_sc = po.dense_ranking(q, V, vis)
        total = min(ref_ids.size, 2_300)
        cur = pvs.pvs_cursor_open(index, q)
        try:
            ids, sc = [], []
            for k in (7, 20, 100, 256, 900, 700, 317):   # past the first horizon
                i, s, _ = pvs.pvs_next(cur, k)
                ids.append(i)
                sc.append(s)
            st = pvs.pvs_cursor_stats(cur)
        finally:
            pvs.pvs_cursor_close(cur)
    finally:
        pvs.pvs_index_free(index)
    ids, sc = np.concatenate(ids), np.concatenate(sc)
    assert ids.size == total == st["emitted"]
    assert np.array_equal(ids, ref_ids[:total])
    assert np.array_equal(sc.view(np.uint32), ref_sc[:total].view(np.uint32))


@pytest.mark.parametrize("pages", [1, 4])
def test_a_set_read_ahead_is_kept(pages):
    """pvs_cursor_set_readahead bounds what the first pull computes ahead."""
    rng = np.random.default_rng(pages)
    V = _corpus("clusters", 40_001, 96, rng)
    index = pvs.pvs_build(V)
    try:
        cur = pvs.pvs_cursor_open(index, V[0])
        try:
            pvs.pvs_cursor_set_readahead(cur, pages)
            ids, sc, _ = pvs.pvs_next(cur, 20)
            lo, _ = pvs.pvs_cursor_bounds(cur, 0, V.shape[0])
        finally:
            pvs.pvs_cursor_close(cur)
    finally:
        pvs.pvs_index_free(index)
    assert np.isneginf(lo).sum() == 20 * pages   # delivered, or computed ahead
    ref_ids, ref_sc = po.dense_ranking(V[0], V)
    assert np.array_equal(ids, ref_ids[:20])
    assert np.array_equal(sc.view(np.uint32), ref_sc[:20].view(np.uint32))
