"""A row that misses its interval deep in a list (App. A.1 failure rule) fails the
pull that reaches it, and no page before it (arXiv 2608.07152 Sec. 2.1: what was
delivered stands)."""
import numpy as np
import pytest

import paper_2608_07152_gb300 as pvs
import synth
from oracle import pvs_oracle as po

pytestmark = pytest.mark.gpu


def _tampered(V, row, factor):
    """An index of V with one row's scale made wrong."""
    built = pvs.pvs_build(V)
    try:
        codes, scale, vnorm, enorm = pvs.pvs_index_export(built, 0, V.shape[0])
    finally:
        pvs.pvs_index_free(built)
    scale[row] *= np.float32(factor)
    return pvs.pvs_index_import(V, codes, scale, vnorm, enorm)


@pytest.mark.parametrize("rank,factor", [(60, 0.9), (250, 0.9), (310, 0.9), (100, 1.3)])
def test_a_violation_past_the_first_page_fails_where_it_is_read(rank, factor):
    n, dim = 20_000, 128
    V = synth.unit_normal(n, dim, seed=31).numpy()
    q = synth.unit_normal(1, dim, seed=32).numpy()[0]
    ref_ids, ref_sc = po.dense_ranking(q, V)
    row = int(ref_ids[rank])
    index = _tampered(V, row, factor)
    try:
        cur = pvs.pvs_cursor_open(index, q)
        try:
            lo, hi = pvs.pvs_cursor_bounds(cur, 0, n)
            # the interval misses the score, and the row is in the first set of 312
            assert not lo[row] <= ref_sc[rank] <= hi[row] and hi[row] > np.sort(lo)[-312]
            got = 0
            with pytest.raises(pvs.PvsError) as e:
                while got < 2 * rank:
                    ids, sc, _ = pvs.pvs_next(cur, 20)
                    assert np.array_equal(ids, ref_ids[got:got + 20])
                    assert np.array_equal(sc.view(np.uint32),
                                          ref_sc[got:got + 20].view(np.uint32))
                    got += 20
                    assert pvs.pvs_cursor_stats(cur)["state"] == pvs.PVS_OK
            # every page above the row, and none with it
            assert e.value.status == pvs.PVS_ERR_INTERVAL and got == rank // 20 * 20
            with pytest.raises(pvs.PvsError) as e:
                pvs.pvs_next(cur, 20)
            assert e.value.status == pvs.PVS_ERR_FAILED
        finally:
            pvs.pvs_cursor_close(cur)
    finally:
        pvs.pvs_index_free(index)


def test_other_calls_fail_after_the_ranks_above_a_violation():
    n, dim, rank = 20_000, 128, 100
    V = synth.unit_normal(n, dim, seed=33).numpy()
    q = synth.unit_normal(1, dim, seed=34).numpy()[0]
    ref_ids, _ = po.dense_ranking(q, V)
    index = _tampered(V, int(ref_ids[rank]), 1.3)
    try:
        import torch
        out_i = torch.zeros(rank, dtype=torch.int64, device="cuda")
        out_s = torch.zeros(rank, device="cuda")
        for call in ("device", "batch", "past"):
            cur = pvs.pvs_cursor_open(index, q)
            try:
                ids, _, _ = pvs.pvs_next(cur, 20)
                if call == "device":   # the rest of the ranks above it, then a pull
                    pvs.pvs_next_device(cur, rank - 20, out_i, out_s)
                    pvs.pvs_cursor_sync(cur)
                    ids = np.concatenate([ids, out_i[:rank - 20].cpu().numpy()])
                    with pytest.raises(pvs.PvsError) as e:
                        pvs.pvs_next_device(cur, 1, out_i, out_s)
                elif call == "batch":
                    more, _, _ = pvs.pvs_next_batch([cur], rank - 20)
                    ids = np.concatenate([ids, more[0]])
                    with pytest.raises(pvs.PvsError) as e:
                        pvs.pvs_next_batch([cur], 1)
                else:
                    with pytest.raises(pvs.PvsError) as e:
                        pvs.pvs_next(cur, rank)
                assert e.value.status == pvs.PVS_ERR_INTERVAL
                assert np.array_equal(ids, ref_ids[:ids.size])
            finally:
                pvs.pvs_cursor_close(cur)
    finally:
        pvs.pvs_index_free(index)
