"""Rings whose buffers two consumer groups take in turn (csrc/ring_turns.h), at
depths that are odd: over many tiles, several passes at once, the bounds equal
the single-query pass's bit for bit (arXiv 2608.07152 Sec. 2.3.1, App. A.1)."""
import numpy as np
import pytest
import torch

import paper_2608_07152_gb300 as pvs

pytestmark = pytest.mark.gpu


def _bounds(cur, n):
    lo, hi = pvs.pvs_cursor_bounds(cur, 0, n)
    return lo.view(np.uint32), hi.view(np.uint32)


@pytest.mark.parametrize("n,m,nq", [(200_003, 1000, 8), (64 * 121 + 1, 1024, 5), (130, 1024, 8)])
def test_grouped_pass_of_three_stages_equals_lone_passes(n, m, nq):
    g = torch.Generator(device="cuda").manual_seed(n + m)
    V = torch.randn((n, m), generator=g, device="cuda")
    Q = torch.randn((nq, m), generator=g, device="cuda")
    index = pvs.pvs_build(V)
    try:
        want = []
        for q in Q:
            cur = pvs.pvs_cursor_open(index, q)
            try:
                want.append(_bounds(cur, n))
            finally:
                pvs.pvs_cursor_close(cur)
        streams = [torch.cuda.Stream() for _ in range(4)]
        for _ in range(5):   # four groups in flight, new cursors each time
            groups = [pvs.pvs_cursor_open_group(index, Q, pass_stream=s) for s in streams]
            try:
                for cursors in groups:
                    for cur, (lo, hi) in zip(cursors, want):
                        got = _bounds(cur, n)
                        assert np.array_equal(got[0], lo) and np.array_equal(got[1], hi)
            finally:
                for cursors in groups:
                    for cur in cursors:
                        pvs.pvs_cursor_close(cur)
    finally:
        pvs.pvs_index_free(index)


@pytest.mark.parametrize("n,m,nq", [(200_003, 768, 128), (128 * 305 + 1, 1000, 96), (70_003, 704, 97)])
def test_batched_pass_of_seven_boxes_equals_lone_cursors(n, m, nq):
    g = torch.Generator(device="cuda").manual_seed(n + m)
    V = torch.randn((n, m), generator=g, device="cuda")
    Q = torch.randn((nq, m), generator=g, device="cuda")
    index = pvs.pvs_build(V)
    try:
        want = []
        for q in Q:
            cur = pvs.pvs_cursor_open(index, q)
            try:
                want.append(pvs.pvs_next(cur, 64)[:2])
            finally:
                pvs.pvs_cursor_close(cur)
        for _ in range(5):
            cursors = pvs.pvs_cursor_open_batch(index, Q, 64)
            try:
                ids, sc, _ = pvs.pvs_next_batch(cursors, 64)
            finally:
                pvs.pvs_cursor_close_batch(cursors)
            for i, (wi, ws) in enumerate(want):
                assert np.array_equal(ids[i], wi)
                assert np.array_equal(sc[i].view(np.uint32), ws.view(np.uint32))
    finally:
        pvs.pvs_index_free(index)
