"""The batched pass over the Int8 codes and the executor's blocks that use it
(arXiv 2608.07152 Sec. 2.1, 2.3.1): at the edges of their tiles, query counts
and widths the ranks equal a lone cursor's and the oracle's, bit for bit."""
import numpy as np
import pytest
import torch

import paper_2608_07152_gb300 as pvs
import synth
from oracle import pvs_oracle as po

pytestmark = pytest.mark.gpu


def _mixture(n, m, nq, seed, comps):
    centres = synth.mixture_centres(comps, m, seed=seed, device="cuda")
    return (synth.mixture_rows(n, centres, 0.35, seed=seed + 1),
            synth.mixture_queries(nq, centres, 0.5, seed=seed + 2))


def _lone(index, q, ranks, snap=None):
    cur = pvs.pvs_cursor_open(index, q, snap)
    try:
        return pvs.pvs_next(cur, ranks)[:2]
    finally:
        pvs.pvs_cursor_close(cur)


def _same(a_ids, a_sc, b_ids, b_sc):
    assert np.array_equal(a_ids, b_ids)
    assert np.array_equal(a_sc.view(np.uint32), b_sc.view(np.uint32))


# widths: the narrowest and widest of the streaming pass, a half box at the
# row's end (64 mod 128), and one past either end (the bf16 pass); query
# counts around a chunk (32), a pass (128; 96 from 769 dimensions) and the batch
@pytest.mark.parametrize("n,m,nq", [
    (129, 128, 3), (2_049, 65, 33), (10_000, 192, 128), (9_999, 448, 129), (70_001, 300, 97),
    (20_011, 768, 256), (12_345, 832, 96), (12_345, 1024, 193), (5_001, 64, 40), (5_001, 1100, 40)])
def test_batched_ranks_equal_lone_cursors(n, m, nq):
    V, Q = _mixture(n, m, nq, seed=n + m, comps=max(2, n // 300))
    index = pvs.pvs_build(V)
    horizon = min(n, 60)
    try:
        cursors = pvs.pvs_cursor_open_batch(index, Q, horizon)
        try:
            pages = [pvs.pvs_next_batch(cursors, horizon // 3) for _ in range(3)]
        finally:
            pvs.pvs_cursor_close_batch(cursors)
        ids = np.concatenate([p[0] for p in pages], axis=1)
        sc = np.concatenate([p[1] for p in pages], axis=1)
        for i in range(nq):
            _same(ids[i], sc[i], *_lone(index, Q[i], ids.shape[1]))
    finally:
        pvs.pvs_index_free(index)
    for i in {0, nq // 2, nq - 1}:
        ref_ids, ref_sc = po.dense_ranking(Q[i].cpu().numpy(), V.cpu().numpy())
        _same(ids[i], sc[i], ref_ids[:ids.shape[1]], ref_sc[:ids.shape[1]])


@pytest.mark.parametrize("ranks", [257, 1000, 1024])
def test_deep_batched_pulls_equal_lone_cursors(ranks):
    V, Q = _mixture(150_000, 128, 20, seed=ranks, comps=60)
    index = pvs.pvs_build(V)
    try:
        cursors = pvs.pvs_cursor_open_batch(index, Q, ranks)
        try:
            ids, sc, n_out = pvs.pvs_next_batch(cursors, ranks)
            more, more_sc, _ = pvs.pvs_next_batch(cursors, 300)   # past the horizon
        finally:
            pvs.pvs_cursor_close_batch(cursors)
        for i in range(20):
            want = _lone(index, Q[i], ranks + 300)
            _same(np.concatenate([ids[i], more[i]]), np.concatenate([sc[i], more_sc[i]]), *want)
    finally:
        pvs.pvs_index_free(index)


def _serve(index, Q, ranks, page, on_device, snap=None, group=8):
    ex = pvs.pvs_executor_create(index, 3)
    try:
        pvs.pvs_executor_set_group(ex, group)
        if on_device:
            ids = torch.zeros((Q.shape[0], ranks), dtype=torch.int64, device="cuda")
            sc = torch.zeros((Q.shape[0], ranks), dtype=torch.float32, device="cuda")
            n_out, status, rc = pvs.pvs_executor_run_device(ex, Q, ranks, page, ids, sc, snap)
            ids, sc = ids.cpu().numpy(), sc.cpu().numpy()
        else:
            ids, sc, n_out, status, rc = pvs.pvs_executor_run(ex, Q.cpu().numpy(), ranks, page, snap)
        return ids, sc, n_out, status, rc, pvs.pvs_executor_stats(ex)
    finally:
        pvs.pvs_executor_destroy(ex)


@pytest.mark.parametrize("nq,m,ranks,on_device", [
    (17, 128, 100, False), (128, 96, 1024, True), (130, 384, 333, False), (200, 1024, 64, True)])
def test_blocks_equal_lone_cursors(nq, m, ranks, on_device):
    V, Q = _mixture(70_003, m, nq, seed=nq, comps=50)
    index = pvs.pvs_build(V)
    try:
        ids, sc, n_out, status, rc, st = _serve(index, Q, ranks, 20, on_device)
        assert rc == pvs.PVS_OK and np.all(status == pvs.PVS_OK) and np.all(n_out == ranks)
        assert st["requests"] == nq and st["ranks"] == nq * ranks
        assert st["pages"] == nq * -(-ranks // 20)
        # blocks of at most a pass's queries, not a pass per eight of them
        assert st["interval_passes"] <= -(-nq // (96 if m > 768 else 128)) + 1
        for i in range(0, nq, 7):
            _same(ids[i], sc[i], *_lone(index, Q[i], ranks))
    finally:
        pvs.pvs_index_free(index)


def test_blocks_on_a_snapshot_that_ends_early():
    V, Q = _mixture(70_003, 128, 17, seed=5, comps=50)
    index = pvs.pvs_build(V)
    snap = None
    try:
        keep = np.random.default_rng(0).choice(70_003, 90, replace=False)
        pvs.pvs_tombstone(index, np.setdiff1d(np.arange(70_003), keep))
        snap = pvs.pvs_snapshot_create(index)
        for on_device in (False, True):
            ids, sc, n_out, status, rc, _ = _serve(index, Q, 150, 20, on_device, snap)
            assert rc == pvs.PVS_OK
            assert np.all(status == pvs.PVS_EXHAUSTED) and np.all(n_out == 90)
            assert np.all(ids[:, 90:] == -1) and np.all(np.isnan(sc[:, 90:]))
            for i in range(17):
                _same(ids[i, :90], sc[i, :90], *_lone(index, Q[i], 150, snap))
    finally:
        if snap is not None:
            pvs.pvs_snapshot_free(snap)
        pvs.pvs_index_free(index)


def test_blocks_with_a_bad_query_and_with_sets_past_the_capacity():
    # rows so alike that every interval holds every threshold: no working set
    # fits, and the block's queries share grouped passes
    g = torch.Generator(device="cuda").manual_seed(3)
    base = torch.randn(128, generator=g, device="cuda")
    V = base + 1e-4 * torch.randn((70_003, 128), generator=g, device="cuda")
    Q = base + torch.randn((19, 128), generator=g, device="cuda")
    index = pvs.pvs_build(V)
    try:
        ids, sc, n_out, status, rc, st = _serve(index, Q, 40, 20, False)
        assert rc == pvs.PVS_OK and np.all(n_out == 40)
        assert 1 < st["interval_passes"] <= 1 + 3
        want = [_lone(index, Q[i], 40) for i in range(19)]
        for i in range(19):
            _same(ids[i], sc[i], *want[i])
        bad = Q.clone()
        bad[11, 7] = float("nan")
        ids, sc, n_out, status, rc, st = _serve(index, bad, 40, 20, True)
        assert rc == pvs.PVS_ERR_NONFINITE and status[11] == pvs.PVS_ERR_NONFINITE
        assert n_out[11] == 0 and np.all(ids[11] == -1) and st["failed"] == 1
        for i in range(19):
            if i != 11:
                _same(ids[i], sc[i], *want[i])
    finally:
        pvs.pvs_index_free(index)
