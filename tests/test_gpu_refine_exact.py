"""Exact scores of rows staged in shared memory (two error-free chains an
instruction; arXiv 2608.07152 Sec. 2.1) against the oracle's correctly rounded
ones: dimensions around a lane's float4s and the ring's depths, and rows whose
scores lie on or next to a rounding boundary."""
import numpy as np
import pytest

import paper_2608_07152_gb300 as pvs
from oracle import pvs_oracle as po

pytestmark = pytest.mark.gpu


def _rows(kind, n, m, rng):
    V = rng.standard_normal((n, m)).astype(np.float32)
    if kind == "wide":          # products over 40 binades
        V *= np.exp2(rng.integers(-20, 21, (n, m))).astype(np.float32)
    elif kind == "cancel":      # second half undoes the first up to a last place
        h = m // 2
        V[:, h:2 * h] = -V[:, :h] * np.float32(1 + 2.0 ** -22)
    elif kind == "ties":        # half-way cases and their neighbours 2^-50 away
        V = np.zeros((n, m), np.float32)
        V[:, 0] = 1 + rng.integers(0, 64, n) * np.float32(2.0 ** -23)
        V[:, m // 2] += np.float32(2.0 ** -24)
        V[:, m - 1] += rng.integers(-1, 2, n).astype(np.float32) * np.float32(2.0 ** -50)
    return np.ascontiguousarray(V)


@pytest.mark.parametrize("m", [3, 4, 127, 128, 129, 511, 768, 1_025, 1_700, 3_300, 6_500])
@pytest.mark.parametrize("kind", ["iid", "wide", "cancel", "ties"])
def test_scores_are_correctly_rounded(kind, m):
    n = 333
    rng = np.random.default_rng(m)
    V = _rows(kind, n, m, rng)
    q = np.ones(m, np.float32) if kind == "ties" else rng.standard_normal(m).astype(np.float32)
    if kind == "cancel":
        q[m // 2:2 * (m // 2)] = q[:m // 2]
    index = pvs.pvs_build(V)
    try:
        ref_ids, ref_sc = po.dense_ranking(q, V)
        cur = pvs.pvs_cursor_open(index, q)
        try:
            ids, sc, _ = pvs.pvs_next(cur, n)
            st = pvs.pvs_cursor_stats(cur)
        finally:
            pvs.pvs_cursor_close(cur)
    finally:
        pvs.pvs_index_free(index)
    assert np.array_equal(ids, ref_ids[:n])
    assert sc.tobytes() == ref_sc[:n].astype(np.float32).tobytes()
    if kind == "iid":           # the fast path settles nearly every row
        assert st["exact_fallbacks"] <= 2 + n // 100
