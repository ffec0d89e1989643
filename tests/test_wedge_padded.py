"""Plain counts by tiles (csrc/wedge.cu) of the graphs in test_wedge.py that the bitmaps of
small.cu count by themselves: isolated vertices take them past the bitmaps' largest graph."""
import pytest

import oracle
from test_wedge import GRAPHS

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PAD = 33000  # past 32768 vertices
# the least degree of a tile vertex is 64 below 2^20 vertices, and a graph takes tiles from degree 128 on
TILES = {"degree_128", "one_tile_vertex", "clique_1100", "huge_row", "warp_rows", "rmat13", "empty_run",
         "past_words", "past_words_dense"}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_padded(name):
    import paper_2309_09064_gb300 as tc
    n, s, d = GRAPHS[name]()
    n += PAD
    rp, col = oracle.build_csr(n, s, d)
    ref = oracle.alg4(rp, col, True)
    c = tc.tc_create(0)
    try:
        g = tc.tc_graph_from_csr(c, rp, col)
        for knobs in ({}, {"flat_cap": 96}):
            if knobs:
                tc.tc_set_tuning(c, **knobs)
            T, st = tc.tc_count(c, g)
            assert (T, st["t_same"], st["t_cross"], st["horizontal_edges"], st["levels"]) == \
                (ref["T"], ref["T_same"], ref["T_cross"], ref["E0"], ref["levels"])
            if not knobs:
                assert (st["class_rows"][1] > 0) == (name in TILES) and not any(st["class_rows"][2:])
        tc.tc_graph_free(g)
    finally:
        tc.tc_destroy(c)
