"""Whether a cyclic component is closed in column slices follows from the edges of its
labels: sparse ones are (the level takes one pass), dense ones stay on the row gather,
whose passes repeat.  The choice is made again when another graph is loaded, by every
loader, and counts the edges of the component's labels alone, also past the labels
counted one by one; answers equal the gather's (and the oracle's where it is quick)."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2103_14688_gb300 import workloads as W

pytestmark = pytest.mark.gpu
T = W.TERM


@pytest.fixture(scope="module")
def C():
    from paper_2103_14688_gb300 import cfpq
    cfpq.load()
    return cfpq


def _plus(label=0):
    return W.make_rsm(2, [0], [0, 0], [1], [(0, T, label, 1), (1, T, label, 1)])


def _graph(n, degs, seed, n_labels=None):
    """`degs[l]` random edges of label l a vertex."""
    rng = np.random.Generator(np.random.PCG64(seed))
    m = [int(n * d) for d in degs]
    lbl = np.repeat(np.arange(len(degs)), m)
    o = rng.permutation(len(lbl))
    return W.Graph(n, n_labels or len(degs), rng.integers(0, n, len(lbl), dtype=np.uint32), lbl[o].astype(np.uint32),
                   rng.integers(0, n, len(lbl), dtype=np.uint32))


def _run(ctx, sliced):
    st = ctx.run()
    assert (st.rounds == 2) == sliced, st.rounds
    return ctx.reachable_words(0)


def _sliced(g, label=0, alone=True):
    """The rule for a+: up to 48 Ki distinct edges, or 24 a row while the slices (one a word of a row) are one wave of
    152 SMs, or 5 a row."""
    on = g.lbl == label
    edges = len(np.unique(g.src[on].astype(np.uint64) << np.uint64(16) | g.dst[on]))
    words = (g.n + 127) // 128 * 2
    return edges <= max(48 << 10, g.n * (24 if alone and words <= 152 else 5))


@pytest.mark.parametrize("n,deg", [(300, 200), (300, 100), (1100, 40), (2000, 20), (2000, 40), (8192, 20), (8192, 60),
                                   (11000, 4), (11000, 12), (20000, 3), (20000, 9)])
def test_choice_by_edges(C, n, deg):
    g, r = _graph(n, [deg], n), _plus()
    with C.Context(no_single_cta=1) as ctx, C.Context(no_single_cta=1, max_rounds=1 << 19) as gather:
        for c in (ctx, gather):
            c.load_graph(g)
            c.load_rsm(r)
        words = _run(ctx, _sliced(g))
        gather.run()
        assert (words == gather.reachable_words(0)).all()
    if n <= 2000:
        assert (words == oracle.worklist_words(g, r)[0]).all()


def test_only_the_component_counts(C):
    """Label 1 is dense, label 0 sparse; and labels past those counted one by one share their mean."""
    g = _graph(3000, [2, 60], 1)
    many = _graph(3000, [0.01] * 70 + [40], 2)
    assert [_sliced(g, l) for l in (0, 1)] == [True, False]
    for graph, label, sliced in ((g, 0, True), (g, 1, False), (many, 3, True), (many, 69, True)):
        with C.Context(no_single_cta=1) as ctx:
            ctx.load_graph(graph)
            ctx.load_rsm(_plus(label))
            assert (_run(ctx, sliced) == oracle.worklist_words(graph, _plus(label))[0]).all()


@pytest.mark.parametrize("how", ["host", "device", "noalloc"])
def test_choice_follows_the_graph(C, how):
    import torch
    n, r = 2500, _plus()
    dense, sparse = _graph(n, [90], 1), _graph(n, [2], 2)
    want = [oracle.worklist_words(g, r)[0] for g in (dense, sparse)]
    assert [_sliced(g) for g in (dense, sparse)] == [False, True]
    with C.Context(no_single_cta=1) as ctx:
        ctx.load_graph(dense)
        ctx.load_rsm(r)
        assert (_run(ctx, False) == want[0]).all()
        for k in (1, 0, 1, 1, 0):
            g = (dense, sparse)[k]
            if how == "host":
                ctx.load_graph(g)
            else:
                dev = [torch.from_numpy(a.astype("int32")).cuda() for a in (g.src, g.lbl, g.dst)]
                if how == "device":
                    ctx.load_graph_device(g.n, g.n_terminals, *dev)
                else:
                    p = [ctypes.c_void_p(a.data_ptr()) for a in dev]
                    assert ctx.lib.cfpq_load_graph_device_noalloc(ctx.h, g.n, g.n_terminals, g.m, *p) == C.CFPQ_OK
            assert (_run(ctx, k == 1) == want[k]).all()


def test_batch_and_server(C):
    r = _plus()
    qs = [(_graph(n, [d], n), r) for n, d in ((700, 2), (2500, 90), (8192, 3), (8192, 20))]
    sliced = [_sliced(g, alone=False) for g, _ in qs]
    assert sliced == [True, False, True, False]
    solo = []
    for g, _ in qs:
        with C.Context(no_single_cta=1, max_rounds=1 << 19) as ctx:
            ctx.load_graph(g)
            ctx.load_rsm(r)
            ctx.run()
            solo.append(ctx.reachable_words(0))
    with C.Context() as ctx:
        per, _ = ctx.batch_run(qs)
        for q, st in enumerate(per):
            assert (st.rounds == 2) == sliced[q]
            assert (ctx.batch_reachable_words(q, 0) == solo[q]).all()
    srv = C.Server(qs[1][0], memory_budget=8 << 30)
    t = srv.submit(r)
    while srv.step() != (0, 0):
        pass
    assert (srv.result_words(t, 0) == solo[1]).all()
