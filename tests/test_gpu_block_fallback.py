"""Requests that an executor's block does not serve (arXiv 2608.07152 Sec. 2.1):
a refused query, a cursor's own error and working sets past the pass's capacity
cost the block's other requests nothing, and hold the bounds of every row for
a few groups of requests at a time."""
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


def _serve(index, Q, ranks, page, on_device, workers=1):
    ex = pvs.pvs_executor_create(index, workers)
    try:
        pvs.pvs_executor_set_group(ex, 8)
        if on_device:
            ids = torch.zeros((Q.shape[0], ranks), dtype=torch.int64, device="cuda")
            sc = torch.zeros((Q.shape[0], ranks), dtype=torch.float32, device="cuda")
            n_out, status, rc = pvs.pvs_executor_run_device(ex, Q, ranks, page, ids, sc)
            ids, sc = ids.cpu().numpy(), sc.cpu().numpy()
        else:
            ids, sc, n_out, status, rc = pvs.pvs_executor_run(ex, Q.cpu().numpy(), ranks, page)
        return ids, sc, n_out, status, rc, pvs.pvs_executor_stats(ex)
    finally:
        pvs.pvs_executor_destroy(ex)


def _same(ids, sc, want):
    assert np.array_equal(ids, want[0])
    assert np.array_equal(sc.view(np.uint32), want[1].view(np.uint32))


ROW_STATE = 41   # bytes a row of a cursor's bounds, working set and sort scratch


@pytest.mark.parametrize("workers,on_device", [(1, False), (8, True)])
def test_wide_working_sets_hold_a_few_groups_of_row_state(workers, on_device):
    n, nq, ranks = 400_003, 100, 40
    g = torch.Generator(device="cuda").manual_seed(7)
    base = torch.randn(128, generator=g, device="cuda")
    V = base + 1e-4 * torch.randn((n, 128), generator=g, device="cuda")
    Q = base + torch.randn((nq, 128), generator=g, device="cuda")
    index = pvs.pvs_build(V)
    try:
        want = {i: _lone(index, Q[i], ranks) for i in (0, 50, 99)}
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        ids, sc, n_out, status, rc, st = _serve(index, Q, ranks, 20, on_device, workers)
        grown = before - torch.cuda.mem_get_info()[0]   # (closed cursors keep their buffers)
    finally:
        pvs.pvs_index_free(index)
    assert rc == pvs.PVS_OK and np.all(status == pvs.PVS_OK) and np.all(n_out == ranks)
    assert st["pages"] == nq * 2 and st["interval_passes"] == 1 + -(-nq // 8)
    for i, w in want.items():
        _same(ids[i], sc[i], w)
    # at most four groups of 8, not 100 cursors, and 200 MB for the rest
    assert grown < 8 * min(workers, 4) * ROW_STATE * n * 1.1 + 200e6, grown


def test_repeated_blocks_do_not_spread_row_state_over_the_pool():
    # 40 of 100 requests are wide: their cursors' buffers stay with few cursors
    n, m, nq, ranks = 400_003, 128, 100, 40
    g = torch.Generator(device="cuda").manual_seed(8)
    centres = synth.mixture_centres(150, m, seed=9, device="cuda")
    base = torch.nn.functional.normalize(torch.randn(m, generator=g, device="cuda"), dim=0)
    V = synth.mixture_rows(n, centres, 0.35, seed=10)
    V[::2] = base + 1e-5 * torch.randn(V[::2].shape, generator=g, device="cuda")
    Q = synth.mixture_queries(nq, centres, 0.5, seed=11)
    wide = torch.arange(0, nq, 5, device="cuda").repeat(2)
    wide[nq // 5:] += 2
    Q[wide] = base + 0.02 * torch.randn((wide.numel(), m), generator=g, device="cuda")
    index = pvs.pvs_build(V)
    try:
        want = {i: _lone(index, Q[i], ranks) for i in (0, 1, 2, 3, 95, 99)}
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        for _ in range(6):
            ids, sc, n_out, status, rc, st = _serve(index, Q, ranks, 20, False, 2)
            assert rc == pvs.PVS_OK and np.all(n_out == ranks)
            assert st["interval_passes"] == 1 + -(-wide.numel() // 8)
        grown = before - torch.cuda.mem_get_info()[0]
        for i, w in want.items():
            _same(ids[i], sc[i], w)
    finally:
        pvs.pvs_index_free(index)
    assert grown < 2 * 8 * ROW_STATE * n * 1.1 + 200e6, grown


@pytest.mark.parametrize("on_device", [False, True])
def test_a_refused_query_costs_the_block_no_pass(on_device):
    centres = synth.mixture_centres(50, 128, seed=1, device="cuda")
    V = synth.mixture_rows(70_003, centres, 0.35, seed=2)
    Q = synth.mixture_queries(41, centres, 0.5, seed=3)
    Q[5, 3] = float("inf")
    Q[40, 0] = float("nan")
    index = pvs.pvs_build(V)
    try:
        ids, sc, n_out, status, rc, st = _serve(index, Q, 100, 20, on_device)
        good = [i for i in range(41) if i not in (5, 40)]
        assert rc == pvs.PVS_ERR_NONFINITE and np.all(status[good] == pvs.PVS_OK)
        for i in (5, 40):
            assert status[i] == pvs.PVS_ERR_NONFINITE and n_out[i] == 0
            assert np.all(ids[i] == -1) and np.all(np.isnan(sc[i]))
        assert st["interval_passes"] == 1 and st["failed"] == 2 and st["requests"] == 41
        for i in good:
            _same(ids[i], sc[i], _lone(index, Q[i], 100))
    finally:
        pvs.pvs_index_free(index)


def test_a_cursors_error_fails_its_request_alone():
    n, dim = 70_003, 128
    centres = synth.mixture_centres(50, dim, seed=11, device="cpu")
    V = synth.mixture_rows(n, centres, 0.35, seed=12).numpy()
    Q = synth.mixture_queries(20, centres, 0.5, seed=13).numpy()
    built = pvs.pvs_build(V)
    try:
        codes, scale, vnorm, enorm = pvs.pvs_index_export(built, 0, n)
        top = int(_lone(built, Q[6], 1)[0][0])
        firsts = [_lone(built, q, 100)[0] for q in Q]
    finally:
        pvs.pvs_index_free(built)
    # the first row of request 6, with an interval that misses its score
    scale[top] *= np.float32(1.5)
    index = pvs.pvs_index_import(V, codes, scale, vnorm, enorm)
    try:
        ids, sc, n_out, status, rc, st = _serve(index, torch.from_numpy(Q), 100, 20, False)
        hit = [i for i in range(20) if status[i] != pvs.PVS_OK]
        assert 6 in hit and all(status[i] == pvs.PVS_ERR_INTERVAL for i in hit)
        assert len(hit) < 8 and rc == pvs.PVS_ERR_INTERVAL
        for i in range(20):
            if i not in hit:
                assert n_out[i] == 100 and np.array_equal(ids[i], firsts[i])
        # the block's pass, and a group's (or its cursor's own) for those that failed
        assert st["interval_passes"] <= 1 + max(1, -(-len(hit) // 8))
    finally:
        pvs.pvs_index_free(index)


@pytest.mark.parametrize("on_device", [False, True])
@pytest.mark.parametrize("wide", [False, True])
def test_a_failed_request_keeps_the_ranks_before_its_error(wide, on_device):
    # request 6 meets a row that misses its interval about 200 ranks down; in a
    # block of its own cursors, and among wide working sets served in groups
    n, dim, rank, ranks = 70_003, 128, 200, 400
    g = torch.Generator().manual_seed(21)
    if wide:
        base = torch.randn(dim, generator=g)
        V = (base + 0.02 * torch.randn((n, dim), generator=g)).numpy()
        Q = (base + torch.randn((20, dim), generator=g)).numpy()
    else:
        V = synth.unit_normal(n, dim, seed=22).numpy()
        Q = synth.unit_normal(20, dim, seed=23).numpy()
    built = pvs.pvs_build(V)
    try:
        codes, scale, vnorm, enorm = pvs.pvs_index_export(built, 0, n)
        refs = [_lone(built, q, ranks)[0] for q in Q]
    finally:
        pvs.pvs_index_free(built)
    scale[refs[6][rank]] *= np.float32(1.3)
    index = pvs.pvs_index_import(V, codes, scale, vnorm, enorm)
    try:
        Qt = torch.from_numpy(Q)
        ids, sc, n_out, status, rc, st = _serve(index, Qt.cuda() if on_device else Qt, ranks, 20,
                                                on_device)
        assert status[6] == pvs.PVS_ERR_INTERVAL
        for i in range(20):
            # a lone cursor's pages on this index (queued device pages are void
            # from the last wait on)
            cur, got = pvs.pvs_cursor_open(index, Q[i]), 0
            try:
                while got < ranks:
                    got += pvs.pvs_next(cur, 20)[0].size
            except pvs.PvsError as e:
                assert e.status == status[i] == pvs.PVS_ERR_INTERVAL
            finally:
                pvs.pvs_cursor_close(cur)
            if not on_device or status[i] == pvs.PVS_OK:
                assert n_out[i] == got and np.array_equal(ids[i, :got], refs[i][:got])
        assert wide or on_device or n_out[6] == rank
    finally:
        pvs.pvs_index_free(index)
