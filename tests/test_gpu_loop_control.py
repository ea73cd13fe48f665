"""The loop control that ends every pass, where its launch also decides what the pass
after it extracts: passes without extraction between passes with one, at the row widths
whose extraction launch is several waves of thread blocks (8 and 16 vectors a lane) and
beside narrow queries.  Batches, the host-driven loop, the server and levels that repeat
give the answers, iterations and edge counts of the single query's loop, whose passes
know their level, or the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2103_14688_gb300 import workloads as W

pytestmark = pytest.mark.gpu
T, N = W.TERM, W.NONTERM
WIDE = 19003, 34001  # 297 and 531 words a row: 8 and 16 vectors a lane


@pytest.fixture(scope="module")
def C():
    from paper_2103_14688_gb300 import cfpq
    cfpq.load()
    return cfpq


def _calls():
    """S -> a* (S b | b): the loop state also reads S, so its level repeats in every iteration."""
    return W.make_rsm(4, [0], [0] * 4, [3], [(0, T, 0, 1), (1, T, 0, 1), (1, T, 1, 3), (1, N, 0, 2), (2, T, 1, 3)])


def _sparse(n, seed):
    """Paths of a and b edges, a few chords: small answers, some tens of iterations."""
    rng = np.random.Generator(np.random.PCG64(seed))
    s = np.concatenate([np.flatnonzero(np.arange(n - 1) % 40 != 39), rng.integers(0, n - 1, n // 50)])
    d = s + 1
    d[-(n // 50):] = rng.integers(0, n, n // 50)
    lbl = np.where(s % 40 < 20, 0, 1)
    return W.Graph(n, 2, s.astype(np.uint32), lbl.astype(np.uint32), d.astype(np.uint32))


def _solo(C, g, r, **opts):
    with C.Context(no_single_cta=1, **opts) as ctx:
        ctx.load_graph(g)
        ctx.load_rsm(r)
        st = ctx.run()
        return st.iterations, st.edges_added, [ctx.reachable_words(b) for b in range(r.n_boxes)]


def _same(a, b):
    return a[:2] == b[:2] and all((x == y).all() for x, y in zip(a[2], b[2]))


@pytest.mark.parametrize("n", (2500, 9001) + WIDE)
def test_host_loop(C, n):
    g, r = W.dyck_zipf(n, seed=n)
    assert _same(_solo(C, g, r, loop_mode=C.CFPQ_LOOP_HOST), _solo(C, g, r))


@pytest.mark.parametrize("n", (700, 9001) + WIDE)
def test_repeating_level(C, n):
    g, r = _sparse(n, n), _calls()
    want = oracle.worklist_words(g, r)[0]
    for opts in ({}, {"max_rounds": 1 << 19}, {"loop_mode": C.CFPQ_LOOP_HOST}):
        for _ in range(2):
            assert (_solo(C, g, r, **opts)[2][0] == want).all()


def test_batch(C):
    qs = [W.dyck_zipf(n, seed=n) for n in (300, 1500, 2600) + WIDE] + [W.two_cycles(21, 20), W.two_cycles(8, 9)]
    qs += [(_sparse(n, n), _calls()) for n in (9001, WIDE[1])]
    want = [_solo(C, g, r) for g, r in qs]
    with C.Context() as ctx:
        for _ in range(2):
            per, _ = ctx.batch_run(qs)
            for q, (g, r) in enumerate(qs):
                got = per[q].iterations, per[q].edges_added, [ctx.batch_reachable_words(q, b) for b in range(r.n_boxes)]
                assert _same(got, want[q]), q


def test_server(C):
    g, dyck = W.dyck_zipf(WIDE[0], seed=7)
    pool = [dyck, W.anbn_rsm(), W.abc_dfa_rsm(), _calls()]
    want = [_solo(C, g, r)[2] for r in pool]
    srv = C.Server(g, memory_budget=48 << 30)
    tickets = [srv.submit(r) for r in pool]
    while srv.step() != (0, 0):
        pass
    for t, r, w in zip(tickets, pool, want):
        assert all((srv.result_words(t, b) == w[b]).all() for b in range(r.n_boxes))
