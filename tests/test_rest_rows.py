"""Rows of the pairs that no tile takes (csrc/wedge.cu, k_wedge_rest): cliques and rings, whose
rows are full of triangles, around the lengths where the search of a key changes (rows of more
than 32 keys turn the warp to a table of the row, which takes up to 256), mixed with rows that
have none."""
import numpy as np
import pytest

import graphgen as gg
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PAD = 40000  # isolated vertices: past the bitmaps' largest graph


def ring(n, half):
    i = np.arange(n, dtype=np.uint32)
    return n, np.tile(i, half), np.concatenate([(i + k + 1) % n for k in range(half)]).astype(np.uint32)


def bipartite(n, tuples, seed):
    e = np.random.default_rng(seed).integers(0, n, (2, tuples), dtype=np.uint32)
    return n, e[0] & ~np.uint32(1), e[1] | np.uint32(1)


def past_tiles(k):
    """32 vertices more than tiles hold, all of degree k - 1: cliques whose last ones no tile takes."""
    blocks = (1 << 19) // k + 40
    i, j = np.triu_indices(k, 1)
    off = np.arange(blocks, dtype=np.uint32)[:, None] * np.uint32(k)
    return k * blocks, (i.astype(np.uint32)[None] + off).ravel(), (j.astype(np.uint32)[None] + off).ravel()


GRAPHS = {
    "cliques_33_34": lambda: gg.disjoint_union([gg.complete(33), gg.complete(34)] * 40),
    "cliques_64": lambda: gg.disjoint_union([gg.complete(64)] * 50),
    "cliques_128": lambda: gg.disjoint_union([gg.complete(128)] * 30),
    "ring_120": lambda: ring(5000, 60),
    "mixed": lambda: gg.disjoint_union([gg.complete(k) for k in range(3, 120)] + [bipartite(3000, 90000, 1)]
                                       + [gg.complete(k) for k in range(119, 40, -1)]),
    "past_tiles_257": lambda: past_tiles(257),   # rows of 255, 256 and 257 keys beside each other
    "past_tiles_300": lambda: past_tiles(300),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_rows(name):
    import paper_2309_09064_gb300 as tc
    n, s, d = GRAPHS[name]()
    c = tc.tc_create(0)
    try:
        dev = lambda a: torch.from_numpy(a.astype(np.int32)).cuda()
        g = tc.tc_build_csr(c, n + PAD, dev(s), dev(d))
        if name.startswith("past"):  # cliques: closed forms
            k = int(name[-3:])
            per = np.zeros(n + PAD, np.uint64)
            per[:n] = (k - 1) * (k - 2) // 2
            T = int(per.sum()) // 3
            # every clique is levelled from its first vertex: the others are horizontal
            same, e0 = n // k * ((k - 1) * (k - 2) * (k - 3) // 6), n // k * ((k - 1) * (k - 2) // 2)
        else:
            rp, col = oracle.build_csr(n + PAD, s, d)
            ref = oracle.alg4(rp, col, True)
            _, per = oracle.vertex_counts(rp, col)
            T, same, e0 = ref["T"], ref["T_same"], ref["E0"]
        for _ in range(2):
            got, st = tc.tc_count(c, g)
            assert (got, st["t_same"], st["t_cross"], st["horizontal_edges"]) == (T, same, T - same, e0)
        out = torch.full((n + PAD,), -1, dtype=torch.int64, device="cuda")
        got, st = tc.tc_count_vertices(c, g, out)
        assert got == T and st["t_same"] == same
        assert np.array_equal(out.cpu().numpy().astype(np.uint64), per)
        tc.tc_graph_free(g)
    finally:
        tc.tc_destroy(c)
