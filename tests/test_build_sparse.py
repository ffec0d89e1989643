"""tc_build_csr of few tuples over many vertices (csrc/csr.cu): the limits between the radix
sort and the counting build (2^24 vertices; n / 16 and n / 8192 tuples), and a device
that has room for the sort's scratch only."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def tuples(n, t, seed):
    r = np.random.default_rng(seed)
    s, d = r.integers(0, n, (2, t), dtype=np.uint32)
    s[:4] = [0, n - 1, 5, 5]
    d[:4] = [n - 1, 0, 5, n - 1]
    return s, d


def check(c, n, s, d):
    import paper_2309_09064_gb300 as tc
    g = tc.tc_build_csr(c, n, s, d)
    rp, col = tc.tc_graph_copy_out(c, g)
    keep = s != d
    a, b = s[keep].astype(np.int64), d[keep].astype(np.int64)
    key = np.unique(np.concatenate([a * n + b, b * n + a]))
    assert np.array_equal(col, (key % n).astype(np.uint32))
    assert np.array_equal(rp.astype(np.int64), np.concatenate([[0], np.cumsum(np.bincount(key // n, minlength=n))]))
    assert tc.tc_count(c, g)[0] >= 0  # (uses the build's largest degree)
    tc.tc_graph_free(g)


N = 1 << 24
CASES = [(N - 1, 100000), (N, N // 16), (N, N // 16 + 1), (N, N // 8192), (N, N // 8192 + 1), (N + 77, 4), (N + 77, 300000)]


@pytest.mark.parametrize("n,t", CASES)
def test_limits(n, t):
    import paper_2309_09064_gb300 as tc
    c = tc.tc_create(0)
    try:
        s, d = tuples(n, t, n + t)
        check(c, n, s, d)
        d[t // 2] = n
        with pytest.raises(tc.TcError):
            tc.tc_build_csr(c, n, s, d)
    finally:
        tc.tc_destroy(c)


def test_scratch_that_grows_with_the_vertices():
    """2^23 vertices need 230 MB for the counts; the sort of 5000 tuples next to nothing."""
    import paper_2309_09064_gb300 as tc
    n = 1 << 23
    s, d = tuples(n, 5000, 9)
    torch.cuda.empty_cache()
    c = tc.tc_create(0)
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (180 << 20), dtype=torch.uint8, device="cuda")
    try:
        g = tc.tc_build_csr(c, n, s, d)
        rp, col = tc.tc_graph_copy_out(c, g)
        tc.tc_graph_free(g)
    finally:
        del fill
        torch.cuda.empty_cache()
        tc.tc_destroy(c)
    keep = s != d
    a, b = s[keep].astype(np.int64), d[keep].astype(np.int64)
    key = np.unique(np.concatenate([a * n + b, b * n + a]))
    assert np.array_equal(col, (key % n).astype(np.uint32)) and int(rp[-1]) == len(key)
