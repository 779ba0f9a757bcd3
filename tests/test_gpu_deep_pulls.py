"""Pulls too deep for one launch (arXiv 2608.07152 Sec. 2.1, 2.3.1): the ranks
ordered by counting, and by the radix sort where more keys reach the last
rank's score, equal the oracle's."""
import numpy as np
import pytest

import paper_2608_07152_gb300 as pvs
from oracle import pvs_oracle as po

pytestmark = pytest.mark.gpu


def _corpus(kind, n, m, rng):
    if kind == "tied":          # about n / 6 rows share each score
        return rng.standard_normal((6, m)).astype(np.float32)[rng.integers(0, 6, n)]
    V = rng.standard_normal((n, m)).astype(np.float32)
    if kind == "alike":         # every interval holds every threshold
        V = (V[0] + 1e-3 * V).astype(np.float32)
    return np.ascontiguousarray(V)


# around the deepest pull of one launch (256), of a batch (1,024), and the keys
# ordered by counting (8,192: the ranks asked for, or the ties of the last)
@pytest.mark.parametrize("kind", ["iid", "tied", "alike"])
@pytest.mark.parametrize("depths", [(257, 300, 1_024, 1_025), (8_191, 2, 8_192, 33), (8_193, 9),
                                    (60_001, 9_998, 1)])
def test_deep_pulls_equal_the_oracle(kind, depths):
    n, m = 70_003, 48
    rng = np.random.default_rng(sum(depths))
    V = _corpus(kind, n, m, rng)
    q = rng.standard_normal(m).astype(np.float32)
    ref_ids, ref_sc = po.dense_ranking(q, V)
    index = pvs.pvs_build(V)
    try:
        cur = pvs.pvs_cursor_open(index, q)
        try:
            pvs.pvs_cursor_set_readahead(cur, 1)
            at = 0
            for k in depths:
                ids, sc, _ = pvs.pvs_next(cur, k)
                assert np.array_equal(ids, ref_ids[at:at + k])
                assert np.array_equal(sc.view(np.uint32), ref_sc[at:at + k].view(np.uint32))
                at += k
        finally:
            pvs.pvs_cursor_close(cur)
    finally:
        pvs.pvs_index_free(index)
