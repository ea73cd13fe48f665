"""Reading an answer back: rows with and without a padding word, answers of
one and of several transfer chunks and beyond the size from which the host
pages are touched first, and a memory budget that leaves no room for the
packing scratch.  The query answers the edges of one label, so the expected
words are known."""
import numpy as np
import pytest

from paper_2103_14688_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C():
    from paper_2103_14688_gb300 import cfpq
    cfpq.load()
    return cfpq


RSM = W.make_rsm(2, [0], [0, 0], [1], [(0, W.TERM, 0, 1)])


def _graph_and_words(n, m, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    g = W.Graph(n, 1, rng.integers(0, n, m, dtype=np.uint32), np.zeros(m, dtype=np.uint32),
                rng.integers(0, n, m, dtype=np.uint32))
    want = np.zeros((n, (n + 63) // 64), dtype=np.uint64)
    np.bitwise_or.at(want, (g.src, g.dst >> 6), np.uint64(1) << (g.dst & 63).astype(np.uint64))
    return g, want


# (wn, W): equal at 128, 700, 16384; a padding word at 1, 64, 130, 1950, 33030 (two chunks of 128 MiB)
@pytest.mark.parametrize("n", [1, 64, 128, 130, 700, 1950, 16384, 33030])
def test_words_equal_edges(C, n):
    g, want = _graph_and_words(n, 4 * n, n)
    with C.Context() as ctx:
        ctx.load_graph(g)
        ctx.load_rsm(RSM)
        ctx.run()
        assert (ctx.reachable_words(0) == want).all()


def test_server_words_equal_edges(C):
    g, want = _graph_and_words(1950, 8000, 3)
    srv = C.Server(g)
    t = srv.submit(RSM)
    while srv.step() != (0, 0):
        pass
    assert (srv.result_words(t) == want).all()
    srv.close()


def test_budget_without_room_for_the_scratch(C):
    n = 1950  # the scratch would take 0.48 MB
    g, want = _graph_and_words(n, 8000, 4)
    step = 64 << 10
    for k in range(1, 200):
        with C.Context(memory_budget=k * step) as ctx:
            try:
                ctx.load_graph(g)
                ctx.load_rsm(RSM)
                ctx.run()
            except C.CfpqError as e:
                assert e.status == C.CFPQ_ERR_OUT_OF_MEMORY
                continue
            assert (ctx.reachable_words(0) == want).all()
            return
    raise AssertionError("no budget sufficed")
