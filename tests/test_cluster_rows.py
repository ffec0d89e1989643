"""Cluster BFS (csrc/levels.cu): claimed vertices of long rows are spread over the blocks.

Chains of cliques and of stars, and rings, of degrees around the limits: 32 (kFarRow), 256
(the whole cluster expands a row) and 4096 (a launch ends).  One block that claimed a
whole clique of 200 had more edges than its queue holds, and every second level went to
the host's loop, which shows in the launches."""
import numpy as np
import pytest

import graphgen as gg
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def chain(parts, k, last):
    """`parts` graphs of k vertices in a row, vertex `last` of each joined to vertex 0 of the next."""
    n, s, d = gg.disjoint_union(parts)
    c = np.arange(len(parts) - 1, dtype=np.uint32) * k
    return n, np.concatenate([s, c + last]).astype(np.uint32), np.concatenate([d, c + k]).astype(np.uint32)


def ring(n, half):
    i = np.arange(n, dtype=np.uint32)
    return n, np.tile(i, half), np.concatenate([(i + k + 1) % n for k in range(half)]).astype(np.uint32)


GRAPHS = {
    "cliques_32": (lambda: chain([gg.complete(32)] * 300, 32, 31), True),
    "cliques_34": (lambda: chain([gg.complete(34)] * 300, 34, 33), True),
    "cliques_200": (lambda: chain([gg.complete(200)] * 60, 200, 199), True),
    "cliques_300": (lambda: chain([gg.complete(300)] * 20, 300, 299), False),
    "ring_66": (lambda: ring(70001, 33), True),
    "ring_200": (lambda: ring(70001, 100), True),
    "stars_1100": (lambda: chain([gg.star(1100)] * 90, 1101, 0), True),
    "stars_4094": (lambda: chain([gg.star(4094)] * 20, 4095, 0), True),
    "stars_4095": (lambda: chain([gg.star(4095)] * 20, 4096, 0), False),
}


@pytest.mark.parametrize("order", ["degree", "id"])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_long_rows(name, order):
    """Levels by the oracle; a level of the host's loop takes four launches or more."""
    import paper_2309_09064_gb300 as tc
    (n, s, d), one_launch = GRAPHS[name][0](), GRAPHS[name][1]
    pad = 70000  # past the size one launch levels whole
    rp, col = oracle.build_csr(n + pad, s, d)
    ref = oracle.alg4(rp, col, order == "degree")
    c = tc.tc_create(0, order=tc.TC_ORDER_DEGREE if order == "degree" else tc.TC_ORDER_ID)
    try:
        g = tc.tc_graph_from_csr(c, rp, col)
        L = torch.full((n + pad,), -7, dtype=torch.int32, device="cuda")
        T, st = tc.tc_count_levels(c, g, L)
        assert np.array_equal(L.cpu().numpy().view(np.uint32), ref["L"])
        assert (T, st["levels"], st["horizontal_edges"]) == (ref["T"], ref["levels"], ref["E0"])
        if one_launch:
            assert st["launches"] < 60  # (every other level by the host's loop: 100 and more)
        tc.tc_graph_free(g)
    finally:
        tc.tc_destroy(c)
