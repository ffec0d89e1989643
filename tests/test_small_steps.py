"""Steps that small graphs take in one launch: ranks by counting (up to 16384
vertices) and by the radix sort's short tiles, and the leftover components in one
block (up to 8192 vertices, none of degree above 256)."""
import numpy as np
import pytest

import graphgen as gg
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def with_rest(parts, hub=4000):
    """A star of `hub` leaves (the first component levelled) beside `parts`."""
    return gg.disjoint_union([gg.star(hub)] + parts)


GRAPHS = {
    "ranks_16384": lambda: gg.er(16384, 60000, 1),
    "ranks_16385": lambda: gg.er(16385, 60000, 2),
    "short_tiles": lambda: gg.er(1 << 19, 1 << 19, 3),
    "long_tiles": lambda: gg.er((1 << 19) + 1, 1 << 19, 4),
    "rest_cycles": lambda: with_rest([gg.cycle(k) for k in range(3, 90)] + [gg.complete(30)] * 3),
    "rest_8192": lambda: with_rest([gg.path(8192)], 9000),
    "rest_8193": lambda: with_rest([gg.path(8193)], 9000),
    "rest_256": lambda: with_rest([gg.star(256)] * 3 + [gg.wheel(40)]),
    "rest_257": lambda: with_rest([gg.star(257)] * 3 + [gg.wheel(40)]),
}


@pytest.mark.parametrize("order", ["degree", "id"])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_small_steps(name, order):
    import paper_2309_09064_gb300 as tc
    n, s, d = GRAPHS[name]()
    pad = 70000 if name.startswith("rest") else 0  # past the size one cluster launch levels whole
    rp, col = oracle.build_csr(n + pad, s, d)
    ref = oracle.alg4(rp, col, order == "degree")
    c = tc.tc_create(0, order=tc.TC_ORDER_DEGREE if order == "degree" else tc.TC_ORDER_ID)
    try:
        g = tc.tc_graph_from_csr(c, rp, col)
        L = torch.full((n + pad,), -7, dtype=torch.int32, device="cuda")
        T, st = tc.tc_count_levels(c, g, L)
        assert np.array_equal(L.cpu().numpy().view(np.uint32), ref["L"])
        assert (T, st["t_same"], st["levels"], st["horizontal_edges"]) == \
            (ref["T"], ref["T_same"], ref["levels"], ref["E0"])
        tc.tc_graph_free(g)
    finally:
        tc.tc_destroy(c)
