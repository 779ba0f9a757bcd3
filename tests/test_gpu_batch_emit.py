"""The emission of batched pulls past one candidate per thread (arXiv
2608.07152 Sec. 2.1, 2.3.1): ranks by score bins, and the sort where ties or an
outlier crowd a bin, equal the oracle's."""
import numpy as np
import pytest

import paper_2608_07152_gb300 as pvs
from oracle import pvs_oracle as po

pytestmark = pytest.mark.gpu


# candidates around a CTA's threads (512) and its keys (2,048), bins around the
# most compared within one (256)
@pytest.mark.parametrize("kind", ["iid", "tied", "outlier", "signs"])
@pytest.mark.parametrize("ranks", [257, 500, 513, 1_000, 1_024])
def test_batched_pulls_of_many_candidates(kind, ranks):
    n, m, nq = 30_011, 128, 9
    rng = np.random.default_rng(ranks)
    V = rng.standard_normal((n, m)).astype(np.float32)
    Q = rng.standard_normal((nq, m)).astype(np.float32)
    if kind == "tied":
        V = V[rng.integers(0, 60, n)]          # about 500 rows per score
    elif kind == "outlier":
        V[n // 2] = 50.0 * Q.sum(axis=0)       # one score far above the rest
    elif kind == "signs":                      # scores of few distinct values
        V, Q = np.sign(V).astype(np.float32), np.sign(Q).astype(np.float32)
    V = np.ascontiguousarray(V)
    index = pvs.pvs_build(V)
    try:
        cursors = pvs.pvs_cursor_open_batch(index, Q, ranks)
        try:
            ids, sc, n_out = pvs.pvs_next_batch(cursors, ranks)
            more, more_sc, _ = pvs.pvs_next_batch(cursors, 600)
        finally:
            pvs.pvs_cursor_close_batch(cursors)
    finally:
        pvs.pvs_index_free(index)
    for i in range(nq):
        ref_ids, ref_sc = po.dense_ranking(Q[i], V)
        for got, got_sc, at in ((ids[i], sc[i], 0), (more[i], more_sc[i], ranks)):
            assert np.array_equal(got, ref_ids[at:at + got.size])
            assert np.array_equal(got_sc.view(np.uint32),
                                  ref_sc[at:at + got.size].view(np.uint32))
