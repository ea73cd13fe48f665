"""Cyclic components closed in column slices: components of one to four states,
several components on one level, states that read nonterminals beside them
(later iterations change the rows they read), long paths (hundreds of
sweeps), hub vertices, duplicate edges, sizes around a thread block and up to the
shared-memory limit.  Answers, iterations and closure rows equal those of a run
whose round cap (never reached) keeps the row gather, and the oracle's answer;
a cap that is reached still ends the run."""
import numpy as np
import pytest

import oracle
from paper_2103_14688_gb300 import workloads as W

pytestmark = pytest.mark.gpu
T, N = W.TERM, W.NONTERM


@pytest.fixture(scope="module")
def C():
    from paper_2103_14688_gb300 import cfpq
    cfpq.load()
    return cfpq


def _rsm(kind):
    if kind == "abc":
        return W.abc_dfa_rsm()
    if kind == "plus":        # a+
        return W.make_rsm(2, [0], [0, 0], [1], [(0, T, 0, 1), (1, T, 0, 1)])
    if kind == "four":        # (a b c a)* with a chord, then b
        return W.make_rsm(5, [0], [0] * 5, [0, 4], [(0, T, 0, 1), (1, T, 1, 2), (2, T, 2, 3), (3, T, 0, 0), (1, T, 0, 0),
                                                    (3, T, 1, 4)])
    if kind == "two loops":   # (a* b c* | c* a)+ : components on several levels, one beside another
        return W.make_rsm(5, [0], [0] * 5, [2, 4], [(0, T, 0, 1), (1, T, 0, 1), (1, T, 1, 2), (2, T, 2, 2), (0, T, 2, 3),
                                                    (3, T, 2, 3), (3, T, 0, 4)])
    # "calls": S -> a* (S b | c): the loop state also reads S; A -> a A | S, called by S
    return W.make_rsm(7, [0, 4], [0, 0, 0, 0, 1, 1, 1], [3, 6],
                      [(0, T, 0, 1), (1, T, 0, 1), (1, T, 2, 3), (0, N, 1, 2), (2, T, 1, 3),
                       (4, T, 0, 5), (5, T, 0, 5), (5, T, 1, 6), (4, N, 0, 6)])


def _graph(kind, n, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    if kind == "path":        # one long path and a few chords
        s, d = np.arange(n - 1), np.arange(1, n)
        s, d = np.concatenate([s, rng.integers(0, n, 5)]), np.concatenate([d, rng.integers(0, n, 5)])
        l = np.where(rng.random(len(s)) < 0.98, 0, rng.integers(0, 3, len(s)))
    else:
        m = 2 * n
        s, d, l = rng.integers(0, n, m), rng.integers(0, n, m), rng.integers(0, 3, m)
        s[: n // 5] = n // 3  # a hub, and duplicate edges
        s[-5:], d[-5:], l[-5:] = s[:5], d[:5], l[:5]
    return W.Graph(n, 3, s.astype(np.uint32), l.astype(np.uint32), d.astype(np.uint32))


def _run(C, g, r, **opts):
    with C.Context(no_single_cta=1, **opts) as ctx:
        ctx.load_graph(g)
        ctx.load_rsm(r)
        st = ctx.run()
        rows = [(s, v) for s in range(r.n_states) for v in (0, 1, g.n // 3, g.n - 1) if v < g.n]
        return st, [ctx.reachable_words(b) for b in range(r.n_boxes)], ctx.closure_rows(rows)


@pytest.mark.parametrize("rsm", ["abc", "plus", "four", "two loops", "calls"])
@pytest.mark.parametrize("graph,n", [("random", 2), ("random", 130), ("random", 1023), ("path", 700), ("random", 4100)])
def test_slices_equal_row_gather(C, rsm, graph, n):
    g, r = _graph(graph, n, n), _rsm(rsm)
    st, words, rows = _run(C, g, r)
    st0, words0, rows0 = _run(C, g, r, max_rounds=1 << 19)
    assert st.iterations == st0.iterations and st.edges_added == st0.edges_added
    assert all((a == b).all() for a, b in zip(words, words0)) and (rows == rows0).all()
    want = oracle.worklist_words(g, r)
    assert all((a == want[b]).all() for b, a in enumerate(words))
    if rsm in ("abc", "plus") and graph == "path":
        assert st.rounds < st0.rounds


# 200 KB: 22755 rows of one state, 11377 of two (the loop (ab)* of "abc")
@pytest.mark.parametrize("rsm,n", [("plus", 22755), ("plus", 22756), ("abc", 11377), ("abc", 11378)])
def test_shared_memory_limit(C, rsm, n):
    g, r = W.random_out_degree_graph(n, 2, 3, n), _rsm(rsm)
    st, words, rows = _run(C, g, r)
    st0, words0, rows0 = _run(C, g, r, max_rounds=1 << 19)
    assert st.iterations == st0.iterations
    assert (words[0] == words0[0]).all() and (rows == rows0).all()


def test_round_cap_still_ends_the_run(C):
    g, r = _graph("path", 700, 1), _rsm("plus")
    with C.Context(no_single_cta=1, max_rounds=3) as ctx:
        ctx.load_graph(g)
        ctx.load_rsm(r)
        with pytest.raises(C.CfpqError) as e:
            ctx.run()
        assert e.value.status == C.CFPQ_ERR_TIMEOUT
