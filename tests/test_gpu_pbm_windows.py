"""PBM pulls whose certified window is larger than what one sort holds, and the
two forms of the range expansion, against the oracle (arXiv 2608.07152
Sec. 2.3.2, App. A.2)."""
import numpy as np
import pytest

import paper_2608_07152_gb300 as pvs
from oracle import pbm_oracle as po

pytestmark = pytest.mark.gpu


def _postings(n_items, n_terms, df, levels, seed):
    """Every term on df random items with impacts of a few levels: flat bounds,
    many exact ties, certified windows of thousands of items."""
    rng = np.random.default_rng(seed)
    docs = [np.sort(rng.choice(n_items, df, replace=False)) for _ in range(n_terms)]
    imps = [1.0 + rng.integers(0, levels, df) for _ in range(n_terms)]
    off = np.arange(n_terms + 1, dtype=np.int64) * df
    return (off, np.concatenate(docs).astype(np.int32),
            np.concatenate(imps).astype(np.float32))


# one term (windows of up to all 40,000 postings), 33 terms (past the warp
# form's 32), ranges of 513 items (past its 512) and a ragged last range
@pytest.mark.parametrize("n_items,n_terms,df,levels,block", [
    (100_000, 1, 40_000, 1, 128), (100_003, 2, 30_000, 3, 128), (50_001, 33, 2_000, 2, 64),
    (50_001, 4, 9_000, 2, 513), (20_000, 32, 700, 5, 512), (9_000, 1, 8_193, 1, 7)])
def test_windows_past_the_sort(n_items, n_terms, df, levels, block):
    off, docs, imps = _postings(n_items, n_terms, df, levels, seed=n_items + n_terms)
    terms = np.arange(n_terms, dtype=np.int32)[::-1].copy()
    weights = np.ones(n_terms, np.float32)
    ref_ids, ref_sc = po.sparse_ranking(terms, weights, off, docs, imps, n_items)
    index = pvs.pbm_build(off, docs, imps, n_items, block)
    try:
        cur = pvs.pbm_cursor_open(index, terms, weights)
        try:
            ids, sc, status = [], [], pvs.PVS_OK
            for k in [20] * 6 + [8_180, 20, 8_192, 33, 8_193, 1, 30_000, 100_000]:
                if status == pvs.PVS_EXHAUSTED:
                    break
                i, s, status = pvs.pbm_next(cur, k)
                ids.append(i)
                sc.append(s)
        finally:
            pvs.pbm_cursor_close(cur)
    finally:
        pvs.pbm_index_free(index)
    ids, sc = np.concatenate(ids), np.concatenate(sc)
    assert status == pvs.PVS_EXHAUSTED or ids.size == ref_ids.size
    assert np.array_equal(ids, ref_ids)
    assert np.array_equal(sc.view(np.uint32), ref_sc.view(np.uint32))
