"""Buffers left by an earlier run: a context that runs graphs of one shape after
another -- full, multiple-source, capped, resumed, column-sharded and single-CTA
runs, in every order -- gives the answers and closure rows of a fresh context."""
import numpy as np
import pytest

from paper_2103_14688_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C():
    from paper_2103_14688_gb300 import cfpq
    cfpq.load()
    return cfpq


def _graphs(kind, n):
    if kind == "rpq":
        return [W.rpq_abc(n=n, out_deg=d, seed=s)[0] for d, s in ((6, 1), (1, 2), (3, 3))], W.abc_dfa_rsm()
    return [W.dyck_zipf(n, seed=s)[0] for s in (1, 2, 3)], W.dyck_rsm(4)


def _read(ctx, r, n):
    rows = [(s, v) for s in range(r.n_states) for v in (0, n // 2, n - 1)]
    return [ctx.reachable_words(b) for b in range(r.n_boxes)], ctx.closure_rows(rows)


def _same(a, b):
    return all((x == y).all() for x, y in zip(a[0], b[0])) and (a[1] == b[1]).all()


@pytest.mark.parametrize("kind,n,opts", [("rpq", 150, {}), ("rpq", 150, {"no_single_cta": 1}), ("rpq", 2500, {}),
                                         ("dyck", 110, {}), ("dyck", 2300, {}), ("dyck", 2300, {"closure_mode": 2}),
                                         ("dyck", 9000, {})])
def test_runs_after_one_another(C, kind, n, opts):
    graphs, r = _graphs(kind, n)
    src = np.array([0, 5, n // 3, n - 1])
    want, want_src = [], []
    for g in graphs:
        with C.Context(**opts) as ctx:
            ctx.load_graph(g)
            ctx.load_rsm(r)
            ctx.run()
            want.append(_read(ctx, r, n))
        with C.Context(**opts) as ctx:
            ctx.load_graph(g)
            ctx.load_rsm(r)
            ctx.run_sources(src)
            want_src.append(_read(ctx, r, n))
    with C.Context(**opts) as ctx:
        ctx.load_graph(graphs[0])
        ctx.load_rsm(r)
        for g, sources in ((0, False), (1, False), (2, True), (1, True), (0, False), (0, True), (2, False), (1, False)):
            ctx.load_graph(graphs[g])
            if sources:
                ctx.run_sources(src)
                assert _same(_read(ctx, r, n), want_src[g])
            else:
                ctx.run()
                assert _same(_read(ctx, r, n), want[g])
        # resumed from the answer of another graph's subset (here: nothing but the answer itself), then plain again
        ctx.set_start(np.stack(want[1][0]))
        ctx.run()
        assert all((a == b).all() for a, b in zip(_read(ctx, r, n)[0], want[1][0]))
        ctx.set_start(None)
        ctx.load_graph(graphs[2])
        ctx.run()
        assert _same(_read(ctx, r, n), want[2])


def test_after_a_capped_run(C):
    g0, r = W.dyck_zipf(2300, seed=5)
    g1, _ = W.dyck_zipf(2300, seed=6)
    with C.Context() as ctx:
        ctx.load_graph(g1)
        ctx.load_rsm(r)
        ctx.run()
        want = _read(ctx, r, 2300)
    with C.Context(max_iterations=60) as ctx:
        ctx.load_graph(g0)
        ctx.load_rsm(r)
        ctx.run()
        ctx.load_graph(g1)
        ctx.run()
        assert _same(_read(ctx, r, 2300), want)
    with C.Context(max_iterations=3) as ctx:
        ctx.load_rsm(r)
        for g in (g0, g1):
            ctx.load_graph(g)
            with pytest.raises(C.CfpqError):
                ctx.run()
            first = [ctx.reachable_words(b) for b in range(r.n_boxes)]
    with C.Context(max_iterations=3) as ctx:
        ctx.load_rsm(r)
        ctx.load_graph(g1)
        with pytest.raises(C.CfpqError):
            ctx.run()
        assert all((a == ctx.reachable_words(b)).all() for b, a in enumerate(first))
