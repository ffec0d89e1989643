"""Graphs of up to 65536 vertices (csrc/small.cu): alone (the same / cross split)
and in a union, with rows at the lane, warp and block limits, rows walked in
slices, ids at the ends of the 16-bit range, and a graph one vertex too large.
Counts are whole numbers: no tolerance."""
import numpy as np
import pytest

import graphgen as gg
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def at_end(n, graph):
    """The graph's vertices as the last of n."""
    k, s, d = graph[:3]
    return n, s + np.uint32(n - k), d + np.uint32(n - k)


GRAPHS = {
    "empty": lambda: (3, np.zeros(0, np.uint32), np.zeros(0, np.uint32)),
    "edge": lambda: gg.path(2),
    "k9": lambda: gg.complete(9),
    "k33": lambda: gg.complete(33),       # degree 32: the last lane row
    "k34": lambda: gg.complete(34),       # degree 33: a warp's
    "k66": lambda: at_end(99, gg.complete(66)),  # |N| to 65: one row in slices
    "k300": lambda: at_end(2000, gg.complete(300)),
    "wheel": lambda: gg.wheel(2051),      # degree above 2048: a block's row
    "bipartite": lambda: gg.complete_bipartite(5, 2049),
    "rmat12": lambda: gg.rmat(12, 20, seed=5)[:3],
    "k70_at_end": lambda: at_end(65536, gg.complete(70)),
    "rmat14": lambda: gg.rmat(14, 30, seed=2)[:3],
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_one_graph(name):
    import paper_2309_09064_gb300 as tc
    rp, col = oracle.build_csr(*GRAPHS[name]())
    ref = oracle.alg4(rp, col, True)
    c = tc.tc_create(0)
    try:
        g = tc.tc_graph_from_csr(c, rp, col)
        T, st = tc.tc_count(c, g)
        assert (T, st["t_same"], st["t_cross"], st["horizontal_edges"]) == (
            ref["T"], ref["T_same"], ref["T_cross"], ref["E0"])
        tc.tc_graph_free(g)
    finally:
        tc.tc_destroy(c)


@pytest.mark.parametrize("extra", [None, 65537])
def test_union(extra):
    """All of them in one batch, in two orders; a larger graph takes the union to the classes."""
    import paper_2309_09064_gb300 as tc
    graphs = [GRAPHS[k]() for k in sorted(GRAPHS)]
    if extra:
        graphs.append(at_end(extra, gg.complete(12)))
    csr = [oracle.build_csr(*g) for g in graphs]
    ref = [oracle.alg4(*x, True)["T"] for x in csr]
    c = tc.tc_create(0)
    try:
        tc.tc_set_tuning(c, batch_small_slots=0)
        gs = [tc.tc_graph_from_csr(c, *x) for x in csr]
        assert list(tc.tc_count_batch(c, gs)) == ref
        assert list(tc.tc_count_batch(c, gs[::-1])) == ref[::-1]
        for g in gs:
            tc.tc_graph_free(g)
    finally:
        tc.tc_destroy(c)


def test_classes_when_the_tiles_scratch_does_not_fit():
    """Device memory for the classes' scratch but not for the tiles': the count takes the classes."""
    import paper_2309_09064_gb300 as tc
    rp, col = oracle.build_csr(*gg.rmat(18, 16, seed=3)[:3])
    want = oracle.alg4(rp, col, True)

    def count(tuned, c):
        if tuned:
            tc.tc_set_tuning(c, flat_cap=96)
        g = tc.tc_graph_from_csr(c, rp, col)
        T, st = tc.tc_count(c, g)
        held = tc.tc_arena_bytes(c)
        tc.tc_graph_free(g)
        assert (T, st["t_same"]) == (want["T"], want["T_same"])
        return held, sum(st["class_rows"][2:]) > 0

    def fresh(tuned):
        c = tc.tc_create(0)
        try:
            return count(tuned, c)
        finally:
            tc.tc_destroy(c)

    (tiles, no), (classes, yes) = fresh(False), fresh(True)  # (an arena holds 9/8 of what a count asks for)
    assert not no and yes and tiles > classes + (16 << 20)
    c = tc.tc_create(0)
    try:
        g = tc.tc_graph_from_csr(c, rp, col)  # (its memory comes before the rest is taken)
        torch.cuda.empty_cache()
        room = (tiles + classes) // 2 * 8 // 9
        fill = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
        try:
            T, st = tc.tc_count(c, g)
        finally:
            del fill
            torch.cuda.empty_cache()
        assert (T, st["t_same"]) == (want["T"], want["T_same"])
        assert sum(st["class_rows"][2:]) > 0
        tc.tc_graph_free(g)
    finally:
        tc.tc_destroy(c)


@pytest.mark.parametrize("form", ["count", "batch"])
def test_threads_with_graphs_of_different_sizes(form):
    """Two contexts count small and large graphs at once: what a launch may use is set for all of them."""
    import threading
    import paper_2309_09064_gb300 as tc
    sizes = [gg.rmat(7, 8, seed=1)[:3], gg.rmat(15, 8, seed=1)[:3]] if form == "batch" else [
        gg.rmat(16, 8, seed=1)[:3], gg.rmat(19, 8, seed=1)[:3]]
    errors = []

    def work(graph):
        c = tc.tc_create(0)
        try:
            rp, col = oracle.build_csr(*graph)
            want = oracle.alg4(rp, col, True)["T"]
            g = tc.tc_graph_from_csr(c, rp, col)
            for _ in range(150):
                got = list(tc.tc_count_batch(c, [g, g])) if form == "batch" else [tc.tc_count(c, g)[0]]
                if set(got) != {want}:
                    errors.append((got, want))
            tc.tc_graph_free(g)
        except Exception as e:  # noqa: BLE001 -- reported by the test's thread
            errors.append(e)
        finally:
            tc.tc_destroy(c)

    threads = [threading.Thread(target=work, args=(x,)) for x in sizes for _ in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
