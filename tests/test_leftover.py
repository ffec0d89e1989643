"""Components beside the first (csrc/levels.cu): which ones one block levels (k_residual)
and which go to the kernels of the host's loop, at the limits of either, and many small
ones in a graph that one cluster launch levels whole."""
import numpy as np
import pytest

import graphgen as gg
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def count(n, s, d):
    import paper_2309_09064_gb300 as tc
    rp, col = oracle.build_csr(n, s, d)
    ref = oracle.alg4(rp, col, True)
    c = tc.tc_create(0)
    try:
        g = tc.tc_graph_from_csr(c, rp, col)
        L = torch.full((n,), -7, dtype=torch.int32, device="cuda")
        T, st = tc.tc_count_levels(c, g, L)
        assert np.array_equal(L.cpu().numpy().view(np.uint32), ref["L"])
        assert (T, st["t_same"], st["levels"], st["horizontal_edges"]) == \
            (ref["T"], ref["T_same"], ref["levels"], ref["E0"])
        tc.tc_graph_free(g)
        return st["launches"]
    finally:
        tc.tc_destroy(c)


def beside(*parts):
    """A star of 4000 leaves (the first component levelled) beside `parts`, past the size levelled whole."""
    n, s, d = gg.disjoint_union([gg.star(4000), *parts])
    return n + 70000, s, d


# leftovers, and whether one block takes them
LEFT = {
    "path_4000": (lambda: [gg.path(4000)], True),               # 7998 slots, two a vertex
    "cycle_8192": (lambda: [gg.cycle(8192)], True),             # 16384 slots
    "slots_4096": (lambda: [gg.complete_bipartite(32, 64)], True),
    "slots_4160": (lambda: [gg.complete_bipartite(32, 65)], False),
    "mean_8": (lambda: [gg.er(2000, 8000, 1)], False),
    "mean_200": (lambda: [gg.gnp(1000, 0.2, 2)], False),
    "triangles": (lambda: [gg.complete(3)] * 1300, True),
}


@pytest.mark.parametrize("name", sorted(LEFT))
def test_leftover(name):
    make, one_block = LEFT[name]
    assert (count(*beside(*make())) <= count(*beside(gg.path(5))) + 2) == one_block


@pytest.mark.parametrize("parts", [1, 2, 3, 40, 900])
def test_many_components_in_a_small_graph(parts):
    """Past the second component the vertices left are levelled together."""
    launches = count(*gg.disjoint_union([gg.er(300, 2000, 3)] + [gg.complete(3)] * parts))
    if parts >= 3:
        assert launches == count(*gg.disjoint_union([gg.er(300, 2000, 3)] + [gg.complete(3)] * 4))
