"""Batched opens and blocks for a page or less (arXiv 2608.07152 Sec. 2.3.1):
their thresholds come from a sample of the corpus, as deeper ones' do, so their
scratch does not grow with rows times queries; the ranks equal a lone
cursor's."""
import numpy as np
import pytest
import torch

import paper_2608_07152_gb300 as pvs
import synth

pytestmark = pytest.mark.gpu


def _lone(index, q, ranks):
    cur = pvs.pvs_cursor_open(index, q)
    try:
        return pvs.pvs_next(cur, ranks)[:2]
    finally:
        pvs.pvs_cursor_close(cur)


def _same(ids, sc, want):
    assert np.array_equal(ids, want[0])
    assert np.array_equal(sc.view(np.uint32), want[1].view(np.uint32))


@pytest.mark.parametrize("n,m,comps", [(200_003, 128, 90), (70_003, 384, 0), (1_000_003, 96, 2000)])
def test_short_blocks_equal_lone_cursors(n, m, comps):
    nq = 40
    if comps:
        centres = synth.mixture_centres(comps, m, seed=n, device="cuda")
        V = synth.mixture_rows(n, centres, 0.35, seed=n + 1)
        Q = synth.mixture_queries(nq, centres, 0.5, seed=n + 2)
    else:
        V = synth.unit_normal(n, m, seed=n, device="cuda")
        Q = synth.unit_normal(nq, m, seed=n + 2, device="cuda")
    index = pvs.pvs_build(V)
    try:
        ex = pvs.pvs_executor_create(index, 2)
        try:
            pvs.pvs_executor_set_group(ex, 8)
            want = [_lone(index, q, 31) for q in Q]
            for ranks in (1, 10, 20, 31):
                ids, sc, n_out, status, rc = pvs.pvs_executor_run(ex, Q.cpu().numpy(), ranks,
                                                                  min(ranks, 10))
                assert rc == pvs.PVS_OK and np.all(status == pvs.PVS_OK)
                for i in range(nq):
                    _same(ids[i], sc[i], [w[:ranks] for w in want[i]])
        finally:
            pvs.pvs_executor_destroy(ex)
        for ranks in (5, 31):   # beyond the horizon too
            cursors = pvs.pvs_cursor_open_batch(index, Q, ranks)
            try:
                ids, sc, _ = pvs.pvs_next_batch(cursors, 31)
            finally:
                pvs.pvs_cursor_close_batch(cursors)
            for i in range(nq):
                _same(ids[i], sc[i], want[i])
    finally:
        pvs.pvs_index_free(index)


def test_short_horizons_need_no_scratch_per_row():
    n, nq = 1_000_003, 128
    centres = synth.mixture_centres(1000, 128, seed=1, device="cuda")
    V = synth.mixture_rows(n, centres, 0.35, seed=2)
    Q = synth.mixture_queries(nq, centres, 0.5, seed=3)
    index = pvs.pvs_build(V)
    try:
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        cursors = pvs.pvs_cursor_open_batch(index, Q, 20)
        pvs.pvs_cursor_close_batch(cursors)
        grown = before - torch.cuda.mem_get_info()[0]   # (the scratch pool keeps its memory)
    finally:
        pvs.pvs_index_free(index)
    # working sets of 8,192 rows a query, twice, are 80 MB; a float a row and query is 512 MB
    assert grown < 250e6, grown
