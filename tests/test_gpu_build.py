"""The row quantizer and the query encoder against the oracle, bit for bit
(arXiv 2608.07152 Sec. 2.3.1, App. A.1), at the edges of their paths: widths
around the kernels' register shapes, quotients at and next to half-integers,
and the rows that leave the float32 arithmetic (subnormal maxima, residuals
or scales) beside rows that do not."""
import numpy as np
import pytest

import paper_2608_07152_gb300 as pvs
from oracle import pvs_oracle as po

pytestmark = pytest.mark.gpu


def _rows(m, rng):
    rows = [np.zeros(m, np.float32)]
    for scale in (1.0, 1e30, 1e-30, 1e-37, 3e-39, 2.0 ** -149):
        rows.append((rng.standard_normal(m) * scale).astype(np.float32))
    rows.append((rng.standard_normal(m) * 10.0 ** rng.uniform(-40, 0, m)).astype(np.float32))
    for top in (127.0, 127.0 * (2.0 - 2.0 ** -22), 1.0, np.float32(1) / 3):
        # (c + 1/2) s and its float32 neighbours, for the row's own scale
        s = np.float32(np.float32(top) / np.float32(127.0))
        half = ((rng.integers(-127, 127, m) + 0.5) * np.float64(s)).astype(np.float32)
        half = np.nextafter(half, (half * rng.integers(0, 3, m)).astype(np.float32))
        half = np.clip(half, -np.float32(top), np.float32(top))
        half[rng.integers(0, m)] = np.float32(top)
        rows.append(half)
    ints = rng.integers(-3, 4, m).astype(np.float32)
    rows.append(ints)
    near_max = (rng.standard_normal(m) * 1e36).astype(np.float32)   # norms near the float32 limit
    rows.append(near_max)
    return np.ascontiguousarray(np.stack(rows))


WIDTHS = [1, 3, 4, 31, 64, 127, 128, 129, 255, 385, 512, 640, 769, 1023, 1024, 1025, 1500]


@pytest.mark.parametrize("m", WIDTHS)
def test_rows_equal_the_oracle_quantizer(m):
    rng = np.random.default_rng(m)
    # enough copies that warps take several rows each, the last batch partial
    V = np.concatenate([_rows(m, rng) for _ in range(3)] +
                       [rng.standard_normal((10_007, m)).astype(np.float32)])
    want = po.quantize(V)
    index = pvs.pvs_build(V)
    try:
        codes, scale, vnorm, enorm = pvs.pvs_index_export(index, 0, V.shape[0])
    finally:
        pvs.pvs_index_free(index)
    assert np.array_equal(codes, want.z)
    for got, ref in ((scale, want.s), (vnorm, want.vnorm), (enorm, want.enorm)):
        assert np.array_equal(got.view(np.uint32), ref.view(np.uint32))


@pytest.mark.parametrize("m", WIDTHS)
def test_query_scalars_equal_the_oracle_encoder(m):
    """The bounds of a few rows hold every scalar of the query's encoding."""
    rng = np.random.default_rng(100 + m)
    V = rng.standard_normal((70, m)).astype(np.float32)
    Z = po.quantize(V)
    index = pvs.pvs_build(V)
    try:
        for q in _rows(m, rng)[:-1]:
            cur = pvs.pvs_cursor_open(index, q)
            try:
                lo, hi = pvs.pvs_cursor_bounds(cur, 0, V.shape[0])
            finally:
                pvs.pvs_cursor_close(cur)
            ref_lo, ref_hi = po.intervals(po.encode_query(q), Z, m)
            assert np.array_equal(lo.view(np.uint32), ref_lo.view(np.uint32))
            assert np.array_equal(hi.view(np.uint32), ref_hi.view(np.uint32))
    finally:
        pvs.pvs_index_free(index)
