"""tc_build_csr with vertices named by very many tuples (csrc/csr.cu): rows whose bitmap lies in
global memory, from 2^17 entries and a sixteenth of the vertices on, 64 of them at most."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def hubs(n, sizes, seed, rest=5000):
    """Vertex i (spread over the ids) has sizes[i] tuples to random vertices; `rest` tuples beside them."""
    r = np.random.default_rng(seed)
    ids = np.sort(r.choice(n, len(sizes), replace=False)).astype(np.uint32)
    s = np.concatenate([np.repeat(ids, sizes), r.integers(0, n, rest, dtype=np.uint32)]).astype(np.uint32)
    d = r.integers(0, n, len(s), dtype=np.uint32)
    turn = r.random(len(s)) < 0.5
    p = r.permutation(len(s))
    return n, np.where(turn, d, s)[p], np.where(turn, s, d)[p]


def star_rows(n, sizes):
    """Rows of exactly these entries: centre i named with leaves of its own (repeated when they run out)."""
    k = len(sizes)
    leaves = np.arange(k, n, dtype=np.uint32)
    per = len(leaves) // k
    s = np.concatenate([np.full(m, i, np.uint32) for i, m in enumerate(sizes)])
    d = np.concatenate([leaves[i * per + np.arange(m) % per] for i, m in enumerate(sizes)]).astype(np.uint32)
    return n, s, d


G = 1 << 17
CASES = {
    "limits": lambda: star_rows(300000, [G - 1, G, G + 1, 9000, 8192] + [8000] * 90),
    "few_tuples": lambda: star_rows(300000, [G - 1, G, G + 1, 9000, 8192]),  # (below 2^20: by blocks alone)
    "one": lambda: hubs(1 << 20, [8 * G], 1),
    "two_ranges": lambda: hubs((1 << 20) + 33, [8 * G, G // 2], 2),
    "sixteenth": lambda: hubs((1 << 22) + 5, [1 << 18, (1 << 18) + 4000, G + 500, 3 << 18], 3),  # n / 16 = 2^18
    "repeats": lambda: hubs(1000, [8 * G, G + 5, 200000], 4),
    "past_64": lambda: hubs(90, [G + 100] * 70, 5),
    "few_vertices": lambda: hubs(5, [900000, 400000, 10], 6),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_build(name):
    import paper_2309_09064_gb300 as tc
    n, s, d = CASES[name]()
    rp, col = oracle.build_csr(n, s, d)
    c = tc.tc_create(0)
    try:
        for _ in range(2):  # (the second time in an arena that holds the first's leavings)
            g = tc.tc_build_csr(c, n, s, d)
            got_rp, got_col = tc.tc_graph_copy_out(c, g)
            assert np.array_equal(got_rp, rp) and np.array_equal(got_col, col)
            tc.tc_graph_free(g)
    finally:
        tc.tc_destroy(c)
