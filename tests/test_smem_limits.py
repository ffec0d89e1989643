"""Shared-memory limits of kernels are the process's: contexts in several threads, whose
launches need different amounts (csrc/graphs.cu by graph size, csrc/isect.cu by tuning)."""
import os
import threading

import pytest

import graphgen as gg
import oracle

torch = pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run(jobs, rounds):
    """One thread per (graph, knobs, batch): all counts right, no call fails."""
    import paper_2309_09064_gb300 as tc
    errors = []

    def work(graph, knobs, batch):
        c = tc.tc_create(0)
        try:
            tc.tc_set_tuning(c, **knobs)
            rp, col = oracle.build_csr(*graph)
            want = oracle.alg4(rp, col, True)["T"]
            g = tc.tc_graph_from_csr(c, rp, col)
            for _ in range(rounds):
                got = list(tc.tc_count_batch(c, [g] * 3)) if batch else [tc.tc_count(c, g)[0]]
                if set(got) != {want}:
                    errors.append((got, want))
            tc.tc_graph_free(g)
        except Exception as e:  # noqa: BLE001 -- reported by the test's thread
            errors.append(e)
        finally:
            tc.tc_destroy(c)

    threads = [threading.Thread(target=work, args=j) for j in jobs for _ in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors


@pytest.mark.gpu
def test_block_per_graph():
    """Bitmaps of 20000 to 65000 vertices."""
    knobs = dict(batch_small_slots=1 << 20)
    run([(gg.er(n, 15000, n), knobs, True) for n in (20000, 50000, 65000)], 60)


@pytest.mark.gpu
def test_tunings():
    """The classes with tables of different sizes."""
    g = gg.rmat(13, 16, seed=1)[:3]
    run([(g, dict(flat_cap=96, warp_cap=256), False), (g, dict(flat_cap=96), False)], 60)


def test_no_limit_of_one_call():
    """Kernels whose launches need different amounts are given all that there is (the window between a
    lower limit and another thread's launch is too short to be met by the tests above every time)."""
    for name in ("graphs.cu", "isect.cu", "small.cu"):
        code = open(os.path.join(ROOT, "paper_2309_09064_gb300", "csrc", name)).read()
        assert "allow_dynamic_smem" in code and "cudaFuncSetAttribute" not in code, name
