"""Which path a count of many vertices of high degree takes (csrc/wedge.cu, k_wedge_estimate).

Uniform graphs of high mean degree are counted by the classes (the tiles took up to
seven times as long, and past ten seconds ended in an error), power laws and cliques
by the tiles.  The statistics tell the path: tc_stats of a count forced to the classes
(any class knob away from its default) equal those of one that took them by itself."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def uniform(n, mean, gen):
    pick = lambda: torch.randint(0, n, (int(mean * n / 2),), generator=gen, device=DEV, dtype=torch.int32)
    return n, pick(), pick()


def skewed(n, mean, gen):
    """Tuples whose ends fall towards the low ids (density x^-2/3)."""
    pick = lambda: (torch.rand(int(mean * n / 2), generator=gen, device=DEV).pow_(3) * n).to(torch.int32).clamp_(max=n - 1)
    return n, pick(), pick()


def cliques(k, blocks):
    i = torch.triu_indices(k, k, 1, device=DEV, dtype=torch.int32)
    off = (torch.arange(blocks, device=DEV, dtype=torch.int32) * k)[:, None]
    return k * blocks, (i[0][None] + off).reshape(-1), (i[1][None] + off).reshape(-1)


CASES = {
    # name: (graph, the classes are taken by default)
    "uniform_1024": (lambda g: uniform(131072, 1024, g), True),
    "uniform_odd": (lambda g: uniform(180001, 700, g), True),
    "uniform_4096": (lambda g: uniform(60000, 4096, g), True),
    "uniform_few_dense": (lambda g: uniform(32736, 1024, g), False),   # the words cover every rank
    "uniform_low": (lambda g: uniform(262144, 64, g), False),          # no vertex of degree 256
    "skewed": (lambda g: skewed(262144, 256, g), False),
    "cliques": (lambda g: cliques(400, 200), False),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_path(name):
    import paper_2309_09064_gb300 as tc
    gen = torch.Generator(device=DEV)
    gen.manual_seed(11)
    n, s, d = CASES[name][0](gen)
    torch.cuda.synchronize()
    runs = []
    for knobs in ({}, {"flat_cap": 96}):
        c = tc.tc_create(0)
        try:
            if knobs:
                tc.tc_set_tuning(c, **knobs)
            g = tc.tc_build_csr(c, n, s, d)
            T, st = tc.tc_count(c, g)
            L = torch.empty(n, dtype=torch.int32, device=DEV)
            T2, st2 = tc.tc_count_levels(c, g, L)
            T3, st3 = tc.tc_count_with_levels(c, g, L)
            per = torch.empty(n, dtype=torch.int64, device=DEV)
            T4, st4 = tc.tc_count_vertices(c, g, per)
            tc.tc_graph_free(g)
        finally:
            tc.tc_destroy(c)
        assert T == T2 == T3 == T4 and int(per.sum()) == 3 * T
        for o in (st2, st3, st4):
            assert all(o[k] == st[k] for k in ("t_same", "t_cross", "horizontal_edges"))
        runs.append((T, st["t_same"], st["t_cross"], st["horizontal_edges"], st["levels"], per))
        runs[-1] += ([list(o["class_rows"]) for o in (st, st2, st3, st4)],)
    assert runs[0][:5] == runs[1][:5] and torch.equal(runs[0][5], runs[1][5])
    assert (runs[0][6] == runs[1][6]) == CASES[name][1]
