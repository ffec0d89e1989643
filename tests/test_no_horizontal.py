"""Graphs without a horizontal edge: every triangle has one, so no pair is tried (csrc/wedge.cu, csrc/small.cu)."""
import numpy as np
import pytest

import graphgen as gg
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def bipartite(n, tuples, seed):
    """Random edges between even and odd ids."""
    r = np.random.default_rng(seed)
    e = r.integers(0, n, (2, tuples), dtype=np.uint32)
    return n, e[0] & ~np.uint32(1), e[1] | np.uint32(1)


def hubs(n, k):
    """Complete bipartite graph of k hubs and n - k leaves."""
    leaf = np.arange(k, n, dtype=np.uint32)
    return n, np.tile(leaf, k), np.repeat(np.arange(k, dtype=np.uint32), n - k)


GRAPHS = {
    "small": lambda: bipartite(3000, 60000, 1),         # bitmaps
    "tiles": lambda: bipartite(40000, 1500000, 2),      # tiles, words past every rank
    "high": lambda: bipartite(36000, 2600000, 3),       # tile vertices past the words
    "rest": lambda: bipartite(100000, 1000000, 4),      # no tiles
    "hubs": lambda: hubs(50000, 12),
    "path": lambda: gg.path(40000),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_no_pair_is_tried(name):
    import paper_2309_09064_gb300 as tc
    n, s, d = GRAPHS[name]()
    rp, col = oracle.build_csr(n, s, d)
    ref = oracle.alg4(rp, col, True)
    c = tc.tc_create(0)
    try:
        g = tc.tc_graph_from_csr(c, rp, col)
        T, st = tc.tc_count(c, g)
        assert (T, st["horizontal_edges"], st["levels"]) == (0, 0, ref["levels"]) and ref["T"] == ref["E0"] == 0
        assert st["probes"] == 0 and not any(st["class_probes"])
        out = torch.full((n,), -1, dtype=torch.int64, device="cuda")
        T, st = tc.tc_count_vertices(c, g, out)
        assert T == 0 and st["probes"] == 0 and not bool(out.any())
        counts = tc.tc_count_batch(c, [g, g])
        assert not counts.any()
        tc.tc_graph_free(g)
    finally:
        tc.tc_destroy(c)


def test_one_horizontal_edge():
    """One triangle in a bipartite graph: the pairs are tried again."""
    import paper_2309_09064_gb300 as tc
    for n, t in ((3000, 60000), (40000, 1500000)):
        _, s, d = bipartite(n, t, 5)
        rp, col = oracle.build_csr(n, s, d)
        hub = int(np.argmax(np.diff(rp)))
        w = col[rp[hub]:rp[hub + 1]][:2]
        rp, col = oracle.build_csr(n, np.append(s, w[0]).astype(np.uint32), np.append(d, w[1]).astype(np.uint32))
        ref = oracle.alg4(rp, col, True)
        assert ref["T"] >= 1
        c = tc.tc_create(0)
        try:
            g = tc.tc_graph_from_csr(c, rp, col)
            T, st = tc.tc_count(c, g)
            assert (T, st["t_same"], st["t_cross"], st["horizontal_edges"]) == \
                (ref["T"], ref["T_same"], ref["T_cross"], ref["E0"])
            tc.tc_graph_free(g)
        finally:
            tc.tc_destroy(c)
