"""The wedge path (csrc/wedge.cu): the plain count under the degree order.

Graphs sit on the edges of its cases -- the tile degree (128), tiles of 32
vertices, rows of one lane / one warp / one block, rows of more than 1024
neighbours that precede, ranks past the 32736 a tile's words cover -- and every
count is compared with the oracle's and with the class kernels' (any class knob
set away from its default selects those)."""
import numpy as np
import pytest

import graphgen as gg
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tc():
    import paper_2309_09064_gb300 as m
    return m


def join(*graphs):
    """Union of tuple graphs on the same vertices."""
    return (max(g[0] for g in graphs), np.concatenate([g[1] for g in graphs]).astype(np.uint32),
            np.concatenate([g[2] for g in graphs]).astype(np.uint32))


def hub_and_clique(leaves, k):
    """A star of `leaves` leaves whose first k leaves form a clique with its centre."""
    c = gg.complete(k + 1)
    return join(gg.star(leaves), c)


def dense_blocks(blocks, k, seed):
    """Cliques of k vertices, chained by a few random edges (many vertices of degree k - 1)."""
    n, s, d = gg.disjoint_union([gg.complete(k)] * blocks)
    r = np.random.default_rng(seed)
    e = r.integers(0, n, (2, n // 4), dtype=np.uint32)
    return n, np.concatenate([s, e[0]]).astype(np.uint32), np.concatenate([d, e[1]]).astype(np.uint32)


GRAPHS = {
    "degree_127": lambda: gg.complete(128),          # no vertex reaches the tile degree
    "degree_128": lambda: gg.complete(129),          # all do: five tiles, the last with one vertex
    "one_tile_vertex": lambda: hub_and_clique(128, 5),
    "clique_1100": lambda: gg.complete(1100),        # rows of more than 1024 keys: sorted by a block
    "huge_row": lambda: hub_and_clique(9000, 200),   # a row of degree above 8192
    "lane_rows": lambda: dense_blocks(40, 32, 1),    # rows of at most 32 neighbours, no tiles
    "warp_rows": lambda: dense_blocks(30, 140, 2),
    "past_words": lambda: gg.er(40000, 40000 * 70, 3),  # ranks past 32736 in the tiles (mean degree 140)
    "past_words_dense": lambda: dense_blocks(260, 140, 4),  # 36400 tile vertices, triangles among the last ones
    "rmat13": lambda: gg.rmat(13, 24, seed=7),
    "empty_run": lambda: join((200000, np.zeros(0, np.uint32), np.zeros(0, np.uint32)), gg.complete(300)),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_wedge_counts(tc, name):
    n, s, d = GRAPHS[name]()
    rp, col = oracle.build_csr(n, s, d)
    ref = oracle.alg4(rp, col, True)
    c = tc.tc_create(0)
    try:
        g = tc.tc_graph_from_csr(c, rp, col)
        want = (ref["T"], ref["T_same"], ref["T_cross"], ref["E0"], ref["levels"])
        for knobs in ({}, {}, {"flat_cap": 96}):  # twice the wedge path, then the class kernels
            if knobs:
                tc.tc_set_tuning(c, **knobs)
            T, st = tc.tc_count(c, g)
            assert (T, st["t_same"], st["t_cross"], st["horizontal_edges"], st["levels"]) == want
        tc.tc_graph_free(g)
    finally:
        tc.tc_destroy(c)


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_wedge_vertex_counts(tc, name):
    """Per-vertex counts by tiles: every vertex's triangles, element by element."""
    n, s, d = GRAPHS[name]()
    rp, col = oracle.build_csr(n, s, d)
    _, want = oracle.vertex_counts(rp, col)
    c = tc.tc_create(0)
    try:
        g = tc.tc_graph_from_csr(c, rp, col)
        out = torch.full((n,), -1, dtype=torch.int64, device="cuda")
        T, _ = tc.tc_count_vertices(c, g, out)
        assert np.array_equal(out.cpu().numpy().astype(np.uint64), want) and 3 * T == int(want.sum())
        tc.tc_graph_free(g)
    finally:
        tc.tc_destroy(c)
