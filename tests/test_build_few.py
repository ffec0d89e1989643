"""tc_build_csr of many tuples over few vertices (csrc/csr.cu, k_count_few): the limits of that
count (8192 vertices, 2^16 tuples, 16 a vertex), tiles of 8192 tuples, loops, repeats, bad ids;
and rows past 1024 entries of up to 16384 vertices, which go through bitmaps."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [(1, 70000), (2, 65536), (3, 65535), (5, 65537), (33, 8192 * 9), (1000, 8192 * 9 + 1), (4096, 65536),
         (4097, 65536), (8191, 140001), (8192, 131072), (8192, 131071), (8193, 140000), (700, 3000000),
         (40, 20500), (41, 20900), (16384, 9000000), (16385, 9000000)]


@pytest.mark.parametrize("n,t", CASES)
def test_build(n, t):
    import paper_2309_09064_gb300 as tc
    r = np.random.default_rng(n + t)
    s, d = r.integers(0, n, (2, t), dtype=np.uint32)
    d[::7] = s[::7]            # loops
    s[1:3000] = n - 1          # a run of one vertex
    rp, col = oracle.build_csr(n, s, d)
    c = tc.tc_create(0)
    try:
        g = tc.tc_build_csr(c, n, s, d)
        got_rp, got_col = tc.tc_graph_copy_out(c, g)
        assert np.array_equal(got_rp, rp) and np.array_equal(got_col, col)
        tc.tc_graph_free(g)
        for at in (0, t // 2, t - 1):
            bad = d.copy()
            bad[at] = n if at else 0xFFFFFFFF
            with pytest.raises(tc.TcError):
                tc.tc_build_csr(c, n, s, bad)
            with pytest.raises(tc.TcError):
                tc.tc_build_csr(c, n, bad, s)
    finally:
        tc.tc_destroy(c)
