"""BFS levels from the cluster kernel (csrc/levels.cu): long paths, hubs expanded
by the whole cluster or handed back, queues that overflow, and more components
than one launch roots.  Every level is compared with the oracle's."""
import numpy as np
import pytest

import graphgen as gg
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def chain_of_stars(stars, leaves):
    """Star centres in a path, `leaves` leaves each."""
    n, s, d = gg.disjoint_union([gg.star(leaves)] * stars)
    c = np.arange(stars - 1, dtype=np.uint32) * (leaves + 1)
    return n, np.concatenate([s, c]).astype(np.uint32), np.concatenate([d, c + leaves + 1]).astype(np.uint32)


GRAPHS = {
    "path": lambda: gg.path(5000),
    "grid": lambda: gg.grid(7, 3001, 0.3, 4)[:3],
    "hub_257": lambda: chain_of_stars(3, 256),         # degrees around the cluster-wide limit (256)
    "hub_1025": lambda: chain_of_stars(2, 1024),       # and the degree that ends a launch (1024)
    "many_hubs": lambda: gg.rmat(13, 40, seed=3),      # more hubs in a level than the list holds
    "wide": lambda: gg.complete_bipartite(2, 70000),   # a frontier past every queue
    "wide_tree": lambda: gg.random_tree(90000, 5),
    "components": lambda: gg.disjoint_union([gg.path(k % 7 + 2) for k in range(100)]),  # more roots than a launch takes
    "pairs_and_grid": lambda: gg.disjoint_union([gg.path(2)] * 20 + [gg.grid(40, 41, 0.3, 1)[:3]] + [gg.cycle(9)] * 9),
}


@pytest.mark.parametrize("order", ["degree", "id"])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_levels(name, order):
    import paper_2309_09064_gb300 as tc
    n, s, d = GRAPHS[name]()
    rp, col = oracle.build_csr(n, s, d)
    ref = oracle.alg4(rp, col, order == "degree")
    c = tc.tc_create(0, order=tc.TC_ORDER_DEGREE if order == "degree" else tc.TC_ORDER_ID)
    try:
        g = tc.tc_graph_from_csr(c, rp, col)
        L = torch.full((n,), -7, dtype=torch.int32, device="cuda")
        T, st = tc.tc_count_levels(c, g, L)
        assert np.array_equal(L.cpu().numpy().view(np.uint32), ref["L"])
        assert (T, st["levels"], st["horizontal_edges"]) == (ref["T"], ref["levels"], ref["E0"])
        tc.tc_graph_free(g)
    finally:
        tc.tc_destroy(c)
