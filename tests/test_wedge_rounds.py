"""Tiles whose high keys take several rounds of the hash table (csrc/wedge.cu, k_wedge_high).

A ring of vertices of equal degree fills the first ranks, 32 vertices right
behind it form one tile, and every one of them is joined to `per` ring vertices
of rank 32736 or more: `stride` 2 takes ranks of one parity only, `step` moves
the run of each tile vertex (0: all the same).  Vertices behind the tile close
triangles with it, and vertices of low degree keep the ring's degrees equal."""
import numpy as np
import pytest

import graphgen as gg
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WORDS = 32736   # ranks a tile's words cover
KEYS = 6144     # high keys a round takes
LATER = 20      # vertices behind the tile


def high_tile(ring, half, per, stride, step, spare, odd=0):
    """(n, src, dst); ring vertices have degree 2 * half + spare, the tile's are ring .. ring + 31."""
    ids = np.arange(ring, dtype=np.int64)
    s = [np.repeat(ids, half)]
    d = [(s[0] + np.tile(np.arange(1, half + 1), ring)) % ring]
    used = np.zeros(ring, np.int64)
    for i in range(32):
        w = WORDS + stride * (step * i + np.arange(per + (1 if i < odd else 0)))
        assert w[-1] < ring
        s.append(np.full(len(w), ring + i))
        d.append(w)
        used[w] += 1
        for j in range(LATER):  # a later vertex: the tile vertex and two of its ring vertices
            v = ring + 32 + j
            two = w[[2 * j, 2 * j + 1]]
            if step == 0:       # (all tile vertices share their run: joined once)
                two = two if i == 0 else two[:0]
            s.append(np.full(1 + len(two), v))
            d.append(np.concatenate([[ring + i], two]))
            used[two] += 1
    assert used.max() <= spare
    at = np.repeat(ids, spare - used)
    fill = -(-len(at) // 50)  # at most 50 a vertex
    s.append(at)
    d.append(ring + 32 + LATER + np.arange(len(at)) % fill)
    n = ring + 32 + LATER + fill
    return n, np.concatenate(s).astype(np.uint32), np.concatenate(d).astype(np.uint32)


CASES = {
    "one_parity": (52000, 160, 300, 2, 300, 3),      # 9600 keys, all of even rank
    "three_rounds": (33600, 230, 420, 1, 12, 40),    # 13440 keys of 792 ranks
    "same_run": (33600, 230, 430, 2, 0, 40),         # every key 32 times
    "full_round": (39000, 110, 192, 1, 192, 3),      # 6144 keys
    "one_key_more": (39000, 110, 192, 1, 192, 3, 1),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_rounds(name):
    import paper_2309_09064_gb300 as tc
    case = CASES[name]
    ring = case[0] - case[0] % 32
    n, s, d = high_tile(ring, *case[1:])
    rp, col = oracle.build_csr(n, s, d)
    deg = np.diff(rp).astype(np.int64)
    order = np.lexsort((np.arange(n), -deg))
    assert np.array_equal(order[:ring + 32], np.arange(ring + 32))  # the ranks the construction is about
    keys = sum(int((col[rp[u]:rp[u + 1]] < u).sum() - (col[rp[u]:rp[u + 1]] < WORDS).sum()) for u in range(ring, ring + 32))
    assert keys == 32 * case[2] + (case[6] if len(case) > 6 else 0)
    ref = oracle.alg4(rp, col, True)
    _, per_vertex = oracle.vertex_counts(rp, col)
    c = tc.tc_create(0)
    try:
        g = tc.tc_graph_from_csr(c, rp, col)
        want = (ref["T"], ref["T_same"], ref["T_cross"], ref["E0"], ref["levels"])
        T, st = tc.tc_count(c, g)
        assert (T, st["t_same"], st["t_cross"], st["horizontal_edges"], st["levels"]) == want
        out = torch.full((n,), -1, dtype=torch.int64, device="cuda")
        T, _ = tc.tc_count_vertices(c, g, out)
        assert T == ref["T"] and np.array_equal(out.cpu().numpy().astype(np.uint64), per_vertex)
        tc.tc_graph_free(g)
    finally:
        tc.tc_destroy(c)
