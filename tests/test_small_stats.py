"""Statistics of the counts by bitmaps (csrc/small.cu): tasks, probes and bytes by their definition."""
import numpy as np
import pytest

import graphgen as gg
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GRAPHS = {
    "rmat10": lambda: gg.rmat(10, 16, seed=2)[:3],
    "rmat13": lambda: gg.rmat(13, 20, seed=3)[:3],
    "clique_65": lambda: gg.complete(65),
    "clique_66": lambda: gg.complete(66),      # rows of 65 earlier neighbours: two tasks
    "bipartite": lambda: gg.complete_bipartite(30, 40),
    "star": lambda: gg.star(50),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_class_statistics(name):
    import paper_2309_09064_gb300 as tc
    n, s, d = GRAPHS[name]()
    n += 2000  # (a mean degree the bitmaps take)
    rp, col = oracle.build_csr(n, s, d)
    deg = np.diff(rp).astype(np.int64)
    order = np.lexsort((np.arange(n), -deg))
    rank = np.empty(n, np.int64)
    rank[order] = np.arange(n)
    src = np.repeat(np.arange(n), deg)
    before = rank[col] < rank[src]
    size = np.bincount(src[before], minlength=n)          # |N(v)|
    size[deg < 2] = 0
    rows = size >= 2
    tasks = np.where(size > 64, -(-size // 64), rows.astype(np.int64))
    probes = np.bincount(src[before], weights=size[col[before]], minlength=n).astype(np.int64)
    c = tc.tc_create(0)
    try:
        g = tc.tc_graph_from_csr(c, rp, col)
        _, st = tc.tc_count(c, g)
        tc.tc_graph_free(g)
    finally:
        tc.tc_destroy(c)
    if st["horizontal_edges"] == 0:
        assert not any(st["class_rows"]) and not any(st["class_bytes"]) and st["probes"] == 0
        return
    assert list(st["class_rows"]) == [int(tasks.sum()), 0, 0, 0]
    assert list(st["class_probes"]) == [int(probes[rows].sum()), 0, 0, 0]
    assert list(st["class_bytes"]) == [2 * int((tasks * size)[rows].sum() + probes[rows].sum()), 0, 0, 0]
