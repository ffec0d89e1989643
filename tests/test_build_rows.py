"""tc_build_csr by counting (csrc/csr.cu): rows on the edges of the lane (32),
warp (256, 1024), block (8192) and bitmap sizes, a hub named by most tuples,
vertices past one bitmap range (2^20 ids), heavy repeats, loops, bad ids."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def stars(sizes, spare=0):
    """Disjoint stars of the given sizes, vertex 0 of each its centre; `spare` isolated vertices after them."""
    n, s, d = gg.disjoint_union([gg.star(k) for k in sizes])
    return n + spare, s, d


def shuffled(graph, seed, spread=None):
    """The tuples in another order, each turned round at random, ids spread over `spread` vertices."""
    n, s, d = graph
    r = np.random.default_rng(seed)
    if spread:
        ids = np.sort(r.choice(spread, n, replace=False)).astype(np.uint32)
        s, d, n = ids[s], ids[d], spread
    p = r.permutation(len(s))
    turn = r.random(len(s)) < 0.5
    return n, np.where(turn, d, s)[p], np.where(turn, s, d)[p]


GRAPHS = {
    "row_sizes": lambda: shuffled(stars([1, 31, 32, 33, 64, 65, 255, 256, 257, 512, 513, 1023, 1024, 1025]), 1),
    "block_sizes": lambda: shuffled(stars([2048, 4095, 4097, 8191, 8192, 8193, 20000], spare=3000), 2),
    "past_a_range": lambda: shuffled(stars([9000, 30000, 5]), 3, spread=(1 << 21) + 77),
    "one_hub": lambda: gg.star(300000),
    "repeats": lambda: gg.with_noise(shuffled(gg.rmat(11, 30, seed=5), 4), 5, dup_frac=1.0, loop_frac=0.5),
    "complete": lambda: shuffled(gg.complete(1200), 6),
    "pairs": lambda: (5, np.array([3, 3, 3, 1, 4], np.uint32), np.array([1, 1, 3, 3, 4], np.uint32)),
    "loops_only": lambda: (40, np.arange(40, dtype=np.uint32), np.arange(40, dtype=np.uint32)),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_build(name):
    import paper_2309_09064_gb300 as tc
    n, s, d = GRAPHS[name]()
    rp, col = oracle.build_csr(n, s, d)
    c = tc.tc_create(0)
    try:
        g = tc.tc_build_csr(c, n, s, d)
        got_rp, got_col = tc.tc_graph_copy_out(c, g)
        assert np.array_equal(got_rp, rp) and np.array_equal(got_col, col)
        assert tc.tc_count(c, g)[0] == oracle.count_definition(rp, col)  # (its largest degree is the build's)
        tc.tc_graph_free(g)
        bad = d.copy()
        bad[len(bad) // 2] = n
        with pytest.raises(tc.TcError):
            tc.tc_build_csr(c, n, s, bad)
    finally:
        tc.tc_destroy(c)
