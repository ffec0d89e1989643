"""Repeated counts where the tiles' scratch does not fit: the arena is made once (csrc/count.cu).

The device has room for the classes' scratch only.  TC_FAIL_ALLOC_AT = k fails the
context's k-th allocation: a later count that allocated again would meet one of them
and leave the arena smaller, or fail."""
import pytest

import graphgen as gg
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_one_arena_for_every_count(monkeypatch):
    import paper_2309_09064_gb300 as tc
    rp, col = oracle.build_csr(*gg.rmat(18, 16, seed=3)[:3])
    T = oracle.alg4(rp, col, True)["T"]

    def arena(**knobs):
        c = tc.tc_create(0)
        try:
            tc.tc_set_tuning(c, **knobs)
            g = tc.tc_graph_from_csr(c, rp, col)
            assert tc.tc_count(c, g)[0] == T
            tc.tc_graph_free(g)
            return tc.tc_arena_bytes(c)
        finally:
            tc.tc_destroy(c)

    tiles, classes = arena(), arena(flat_cap=96)
    room = (classes + tiles * 8 // 9) // 2  # (an arena holds 9/8 of what a count asks for, or just that)
    assert tiles * 8 // 9 > classes + (8 << 20)
    repeats = 0
    for k in range(1, 17):
        monkeypatch.setenv("TC_FAIL_ALLOC_AT", str(k))
        c = tc.tc_create(0)
        fill = None
        try:
            g = tc.tc_graph_from_csr(c, rp, col)
            torch.cuda.empty_cache()
            fill = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
            if tc.tc_count(c, g)[0] == T and tc.tc_arena_bytes(c) >= classes:
                repeats += 1
                for _ in range(4):
                    assert tc.tc_count(c, g)[0] == T
                    assert tc.tc_arena_bytes(c) >= classes
            # with the room back the tiles' arena is had again
            del fill
            fill = None
            torch.cuda.empty_cache()
            tc.tc_count(c, g)
            st = tc.tc_count(c, g)[1]
            assert sum(st["class_rows"][2:]) == 0
            tc.tc_graph_free(g)
        except tc.TcError:
            assert k <= 2  # the injected failure met the graph
        finally:
            del fill
            torch.cuda.empty_cache()
            tc.tc_destroy(c)
    assert repeats >= 8
