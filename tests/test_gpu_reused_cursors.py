"""Closed cursors' buffers serve later cursors of larger snapshots and of other
kinds: a batched open's cursor keeps no bounds of every row, whatever buffers it
was handed (arXiv 2608.07152 Sec. 2.1)."""
import numpy as np
import pytest

import paper_2608_07152_gb300 as pvs
import synth
from oracle import pvs_oracle as po

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("first", [20, 300])   # one cluster's pull, and the deep one
def test_batched_cursors_after_lone_cursors_of_a_smaller_index(first, device):
    import torch
    m = 96
    small = synth.unit_normal(700, m, seed=1).numpy()
    more = synth.unit_normal(60_000, m, seed=2).numpy()
    Q = synth.unit_normal(12, m, seed=3).numpy()
    index = pvs.pvs_build(small)
    try:
        lone = [pvs.pvs_cursor_open(index, q) for q in Q]
        for c in lone:
            pvs.pvs_next(c, 10)
        for c in lone:
            pvs.pvs_cursor_close(c)
        pvs.pvs_append(index, more)
        V = np.concatenate([small, more])
        cursors = pvs.pvs_cursor_open_batch(index, Q, 400)
        try:
            ids = torch.zeros(first, dtype=torch.int64, device="cuda")
            sc = torch.zeros(first, device="cuda")
            for q, c in zip(Q, cursors):
                if device:
                    pvs.pvs_next_device(c, first, ids, sc)
                    pvs.pvs_cursor_sync(c)
                    got = ids.cpu().numpy()
                else:
                    got = pvs.pvs_next(c, first)[0]
                got = np.concatenate([got, pvs.pvs_next(c, 350)[0]])
                assert np.array_equal(got, po.dense_ranking(q, V)[0][:first + 350])
        finally:
            pvs.pvs_cursor_close_batch(cursors)
        # and lone cursors on what the batch left
        for q in Q[:3]:
            c = pvs.pvs_cursor_open(index, q)
            try:
                assert np.array_equal(pvs.pvs_next(c, 50)[0], po.dense_ranking(q, V)[0][:50])
            finally:
                pvs.pvs_cursor_close(c)
    finally:
        pvs.pvs_index_free(index)


def test_a_full_pool_of_batched_cursors_leaves_room_for_lone_ones():
    """After 1,024 batched cursors a lone cursor's buffers are still kept: a second
    one takes no more device memory, and its open waits for no cudaFree."""
    import torch
    n, m = 400_000, 128
    V = synth.unit_normal(n, m, seed=11).numpy()
    Q = synth.unit_normal(256, m, seed=12).numpy()
    index = pvs.pvs_build(V)
    try:
        batches = [pvs.pvs_cursor_open_batch(index, Q, 100) for _ in range(4)]
        for b in batches:
            pvs.pvs_cursor_close_batch(b)

        def free_after_a_lone_cursor():
            c = pvs.pvs_cursor_open(index, Q[0])
            pvs.pvs_next(c, 20)
            pvs.pvs_cursor_close(c)
            torch.cuda.synchronize()
            return torch.cuda.mem_get_info()[0]

        before = torch.cuda.mem_get_info()[0]
        first, second = free_after_a_lone_cursor(), free_after_a_lone_cursor()
        # kept: the bounds of every row (lo, hi), at least
        assert before - first >= 8 * n and second == first
    finally:
        pvs.pvs_index_free(index)
