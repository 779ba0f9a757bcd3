"""Host and device reads of one cursor, mixed (include/pvs.h: pvs_next_device only
queues its copies): ranks computed ahead stay where a queued copy reads them until
it has run."""
import numpy as np
import pytest
import torch

import paper_2608_07152_gb300 as pvs
import synth

pytestmark = pytest.mark.gpu


def _busy(stream):
    """Work that keeps the stream for some tens of milliseconds."""
    with torch.cuda.stream(stream):
        x = torch.ones((4096, 4096), device="cuda")
        for _ in range(40):
            x = (x @ x).clamp_(0.0, 1.0)
    return x


@pytest.mark.parametrize("then", ["next", "batch"])
def test_a_host_read_after_a_queued_device_copy(then):
    n, dim = 30_000, 64
    V = synth.unit_normal(n, dim, seed=1, device="cuda")
    q = synth.unit_normal(1, dim, seed=2, device="cuda")[0]
    index = pvs.pvs_build(V)
    st = torch.cuda.Stream()
    try:
        cur = pvs.pvs_cursor_open(index, q)
        try:
            want = pvs.pvs_next(cur, 900)[0]
        finally:
            pvs.pvs_cursor_close(cur)
        for readahead in (4, None):
            cur = pvs.pvs_cursor_open(index, q)
            try:
                pvs.pvs_cursor_set_stream(cur, st.cuda_stream)
                if readahead:
                    pvs.pvs_cursor_set_readahead(cur, readahead)
                first = pvs.pvs_next(cur, 20)[0]
                ids = torch.zeros(25, dtype=torch.int64, device="cuda")
                sc = torch.zeros(25, device="cuda")
                torch.cuda.synchronize()
                keep = _busy(st)
                pvs.pvs_next_device(cur, 25, ids, sc)   # queued behind it, from ranks ahead
                if then == "next":
                    rest = pvs.pvs_next(cur, 600)[0]
                else:
                    rest = pvs.pvs_next_batch([cur], 600)[0][0]
                torch.cuda.synchronize()
                del keep
                got = np.concatenate([first, ids.cpu().numpy(), rest])
                assert np.array_equal(got, want[:got.size])
            finally:
                pvs.pvs_cursor_close(cur)
    finally:
        pvs.pvs_index_free(index)
