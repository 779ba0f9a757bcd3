"""pvs_batch_bounds shows the pass that serves rows of a width (arXiv 2608.07152
Sec. 2.3.1, App. A.1): over the Int8 codes for 65 .. 1,024 dimensions, over a
bf16 copy of them for others; bounds bit for bit the oracle's, query counts
past one pass, deleted rows, tiles that end early."""
import numpy as np
import pytest
import torch

import paper_2608_07152_gb300 as pvs
import synth
from oracle import pvs_oracle as po

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,nq", [(1_025, 64, 33), (515, 65, 129), (2_001, 704, 130),
                                    (387, 832, 97), (129, 1000, 193), (640, 1100, 40)])
def test_bounds_of_both_passes_bit_exact(n, m, nq):
    V = synth.unit_normal(n, m, seed=n).numpy()
    Q = synth.unit_normal(nq, m, seed=n + 1).numpy()
    dead = np.random.default_rng(n).choice(n, n // 20, replace=False)
    index = pvs.pvs_build(V)
    try:
        pvs.pvs_tombstone(index, dead)
        lo, hi = pvs.pvs_batch_bounds(index, Q)
    finally:
        pvs.pvs_index_free(index)
    Qz = po.quantize(V)
    for qi in sorted({0, 31, 32, 95, 96, 127, 128, nq - 1} & set(range(nq))):
        ref_lo, ref_hi = po.intervals(po.encode_query(Q[qi]), Qz, m)
        ref_lo[dead] = ref_hi[dead] = -np.inf
        assert np.array_equal(lo[qi].view(np.uint32), ref_lo.view(np.uint32)), qi
        assert np.array_equal(hi[qi].view(np.uint32), ref_hi.view(np.uint32)), qi


def test_the_bounds_of_the_streaming_pass_need_no_copy_of_the_codes():
    n, m = 400_000, 256
    V = synth.unit_normal(n, m, seed=3, device="cuda")
    Q = synth.unit_normal(1, m, seed=4, device="cuda")
    index = pvs.pvs_build(V)
    try:
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        pvs.pvs_batch_bounds(index, Q)
        grown = before - torch.cuda.mem_get_info()[0]
    finally:
        pvs.pvs_index_free(index)
    assert grown < n * m, grown   # (a bf16 copy is twice that)
