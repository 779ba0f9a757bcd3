"""Exact rank counts of an EAHR finish (arXiv 2608.07152 Sec. 2.1, 2.2) from
each of their sources: the finer centres kept by the fusion's own pass, the
codes where the pass ran before the fusion, the fp32 rows alone; at widths
around the pass's tiles and the residual level's chunks."""
import numpy as np
import pytest

import paper_2608_07152_gb300 as pvs
import synth
from oracle import pvs_oracle as po
from oracle import rrf_oracle as ro

pytestmark = pytest.mark.gpu


def _tied_mid_sparse(dense_ids, pairs, rng):
    """A sparse list that opens with items B_k of the middle of the dense order
    and has the dense top item A_k at B_k's dense rank: F(A_k) = F(B_k), so
    only exact dense ranks order each pair."""
    n = dense_ids.size
    B = dense_ids[n // 2 - 5 * pairs:n // 2 + 5 * pairs:10][:pairs]
    A = dense_ids[:pairs]
    rank = np.empty(n, np.int64)
    rank[dense_ids] = np.arange(n)
    S = np.full(n, -1, np.int64)
    S[:pairs] = B
    S[rank[B]] = A
    rest = dense_ids[~np.isin(dense_ids, np.concatenate([A, B]))].copy()
    rng.shuffle(rest)
    S[S < 0] = rest
    return S


# m_pad 64, 128 and 768, 1,024 (widths of their own), 320 and 1,536 (a run-time
# width), 1,600 (no staged pass: no centres), 4,224 (no residual codes)
@pytest.mark.parametrize("m", [33, 100, 300, 768, 1_023, 1_500, 1_590, 4_200])
@pytest.mark.parametrize("opened", ["fresh", "scanned", "group"])
@pytest.mark.parametrize("scale", [1.0, 1e-18, 1e17])
def test_exact_ranks_from_every_source(m, opened, scale):
    n, pairs = 6_003, 6
    rng = np.random.default_rng(m)
    V = (synth.unit_normal(n, m, seed=m).numpy() * np.float32(scale)).astype(np.float32)
    V[n // 2] = V[n // 3]                           # a tie, decided by id
    V[n - 1] = 0
    q = (synth.unit_normal(1, m, seed=m + 1).numpy()[0] * np.float32(scale)).astype(np.float32)
    dense_ids, _ = po.dense_ranking(q, V)
    S = _tied_mid_sparse(dense_ids, pairs, rng)
    T = ro.target_topk_large([dense_ids, S], [1, 1], 60, 2 * pairs, ro.NUMERATOR)
    index = pvs.pvs_build(V)
    cursors = []
    try:
        if opened == "group":
            cursors = list(pvs.pvs_cursor_open_group(index, np.stack([q, -q])))
        else:
            cursors = [pvs.pvs_cursor_open(index, q)]
            if opened == "scanned":
                pvs.pvs_cursor_bounds(cursors[0], 0, 1)
        ids, F, st = pvs.eahr_topk(cursors[0], S, policy=pvs.EAHR_POLICY_ADAPTIVE, K=2 * pairs,
                                   k=60, form=pvs.EAHR_NUMERATOR)
    finally:
        for c in cursors:
            pvs.pvs_cursor_close(c)
        pvs.pvs_index_free(index)
    assert ids.tolist() == [x for x, _ in T]
    for (_, f), v in zip(T, F):
        assert np.isnan(v) or v == ro.as_float(f)   # NaN: placed by its bounds alone
    assert st["complete"] in (2, 3)
    if m < 4_000:
        assert st["complete"] == 3
